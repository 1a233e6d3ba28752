"""Performance cases: the calls that users of the solver make, at the sizes and degrees they make them.

A case names one public entry point (`kind`), a jittered Kuhn mesh of the unit cube (`n`^3 hexahedra of
six tets), the degrees `p`, `pt`, and the solver's precision.  The kinds:

  step        one time step from a given state (set_state, step, get_state)
  solve       one pressure solve
  apply       one application of the five-point pressure operator, binary64 vectors
  apply_f32   the same on binary32 vectors (binary32 or bfloat16 blocks): the inner iterations' operator
  rhs         the pressure right-hand side b = D F
  update      the velocity update after a pressure solve
  convection  the convective term
  gnn_grad    loss and gradient of the learned preconditioner over a few training pairs
  gnn_apply   the learned preconditioner applied to one residual

`exact` is the same discretisation written in plain binary64 torch from its definition (orthonormal
Dubiner and Legendre bases, Gram-Schmidt dual basis, collapsed Gauss rules).
"""
import functools
import itertools
import math

import numpy as np
import torch

import paper_1601_07384_gb300 as g

DEV = "cuda"
DT = 0.01                       # time step of the largest workload
HIDDEN, LAYERS = 64, 3          # the learned preconditioner's size


def listed():
    return [
        # the smallest workload: 162 tets, every launch and host check counts
        {"name": "step_tiny", "kind": "step", "n": 3, "p": 1, "pt": 0, "precision": "fp64", "method": "kron_cg",
         "data": "beltrami", "nu": 0.1, "npic": 2, "tol": 1e-12},
        # the chosen solver's time step at the degrees of the largest workload
        {"name": "step_p4", "kind": "step", "n": 12, "p": 4, "pt": 4, "precision": "mixed_f32", "method": "kron_mg",
         "data": "solenoidal", "nu": 1e-3, "npic": 3, "tol": 1e-11},
        # the pressure system of the middle workload's degrees by the chosen solver
        {"name": "solve_mixed", "kind": "solve", "n": 16, "p": 3, "pt": 1, "precision": "mixed_f32",
         "method": "kron_mg", "tol": 1e-11},
        # the paper's solver for p_t = 0: plain conjugate gradients in binary64
        {"name": "solve_cg", "kind": "solve", "n": 8, "p": 2, "pt": 0, "precision": "fp64", "method": "cg",
         "tol": 1e-11},
        # the operator of the plain binary64 solvers (GMRES, CG)
        {"name": "apply_fp64", "kind": "apply", "n": 15, "p": 3, "pt": 0, "precision": "fp64"},
        # the binary64-accurate operator of the outer iterations and residual checks
        {"name": "apply_df32", "kind": "apply", "n": 16, "p": 4, "pt": 4, "precision": "df32"},
        # the inner iterations' operator at the middle workload's full size
        {"name": "apply_f32", "kind": "apply_f32", "n": 24, "p": 3, "pt": 1, "precision": "mixed_f32"},
        # the same with bfloat16 blocks, small and odd
        {"name": "apply_bf16", "kind": "apply_f32", "n": 7, "p": 4, "pt": 2, "precision": "mixed_bf16"},
        # one divergence per Picard iteration and per step (diagnostics), at the largest degrees
        {"name": "rhs", "kind": "rhs", "n": 11, "p": 4, "pt": 4, "precision": "mixed_f32"},
        # one update per Picard iteration, at the degrees of the convergence studies
        {"name": "update", "kind": "update", "n": 15, "p": 2, "pt": 2, "precision": "fp64"},
        # the convective term, at the degrees of the middle workload
        {"name": "convection", "kind": "convection", "n": 13, "p": 3, "pt": 1, "precision": "fp64"},
        # one training batch of the learned preconditioner
        {"name": "gnn_grad", "kind": "gnn_grad", "n": 10, "p": 3, "pt": 1, "precision": "mixed_f32", "bf16": True,
         "pairs": 4},
    ]


# largest n per kind and p: no drawn case costs more than the largest listed one
MOST_N = {"apply": {1: 24, 2: 24, 3: 20, 4: 14}, "apply_f32": {1: 24, 2: 24, 3: 24, 4: 14},
          "rhs": {1: 24, 2: 20, 3: 16, 4: 11}, "update": {1: 24, 2: 20, 3: 16, 4: 11},
          "convection": {1: 24, 2: 18, 3: 14, 4: 9}, "step": {1: 10, 2: 10, 3: 9, 4: 8},
          "solve": {1: 16, 2: 14, 3: 12, 4: 9}, "gnn_grad": {1: 12, 2: 12, 3: 10}, "gnn_apply": {1: 16, 2: 16, 3: 12}}
KINDS = ["step", "solve", "apply", "apply", "apply_f32", "apply_f32", "rhs", "update", "convection", "convection",
         "gnn_grad", "gnn_apply"]


def draw(rng):
    kind = rng.choice(KINDS)
    p = rng.choice(sorted(MOST_N[kind]))
    pt = rng.randint(0, 2 if kind.startswith("gnn") else 4)
    lo, hi = 3, MOST_N[kind][p]
    c = {"kind": kind, "n": min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))), "p": p, "pt": pt}
    if kind == "step":
        c.update(precision="mixed_f32", method="kron_mg", data=rng.choice(["beltrami", "solenoidal"]),
                 nu=rng.choice([1e-1, 1e-2, 1e-3]), npic=rng.choice([2, 3]), tol=1e-11)
    elif kind == "solve":
        prec = rng.choice(["mixed_f32", "mixed_f32", "df32", "fp64"])
        c.update(precision=prec, method=rng.choice(["kron_mg", "kron_pcg"]), tol=1e-11)
    elif kind == "apply":
        c.update(precision=rng.choice(["fp64", "df32"]))
    elif kind == "apply_f32":
        c.update(precision=rng.choice(["mixed_f32", "mixed_bf16"]))
    elif kind.startswith("gnn"):
        c.update(precision="mixed_f32", bf16=rng.random() < 0.7)
        if kind == "gnn_grad":
            c.update(pairs=rng.randint(1, 4))
    else:
        c.update(precision=rng.choice(["fp64", "mixed_f32"]))
    return c


# ------------------------------------------------------------------------------------------------ inputs
def kuhn_mesh(n, seed):
    """n^3 hexahedra x 6 tets of the unit cube, interior vertices moved by up to 0.1 h per coordinate."""
    m, h = n + 1, 1.0 / n
    k, j, i = np.meshgrid(*[np.arange(m)] * 3, indexing="ij")
    ijk = np.stack([i.ravel(), j.ravel(), k.ravel()], 1)
    verts = ijk * h
    inner = np.all((ijk > 0) & (ijk < n), 1)
    verts[inner] += np.random.default_rng(seed).uniform(-0.1 * h, 0.1 * h, (int(inner.sum()), 3))
    k, j, i = np.meshgrid(*[np.arange(n)] * 3, indexing="ij")
    base = np.stack([i.ravel(), j.ravel(), k.ravel()], 1)
    tets = np.empty((n ** 3, 6, 4), np.int64)
    for s, pi in enumerate(itertools.permutations(range(3))):
        o = np.zeros((4, 3), np.int64)
        o[1, pi[0]] = 1
        o[2, list(pi[:2])] = 1
        o[3] = 1
        if np.linalg.det((o[1:] - o[0]).astype(float)) < 0:
            o[[2, 3]] = o[[3, 2]]
        for v in range(4):
            q = base + o[v]
            tets[:, s, v] = q[:, 0] + m * (q[:, 1] + m * q[:, 2])
    return verts, tets.reshape(-1, 4)


def multi_indices(p):
    return [(i, j, n - i - j) for n in range(p + 1) for i in range(n + 1) for j in range(n - i + 1)]


def smooth(lead, case, gen):
    """Random space-time coefficients that fall off with the degree, as those of a resolved field do."""
    deg = torch.tensor([sum(e) for e in multi_indices(case["p"])], dtype=torch.float64, device=DEV)
    time = torch.arange(case["pt"] + 1, dtype=torch.float64, device=DEV)
    scale = 0.5 ** deg[None, :] * 0.3 ** time[:, None]
    return torch.randn(*lead, *scale.shape, dtype=torch.float64, device=DEV, generator=gen) * scale


def solenoidal(seed):
    """64 seeded Fourier modes of curl(b Psi) with |v| up to about 0.1, no slip on the walls."""
    r = np.random.default_rng(seed)
    k = r.integers(-4, 5, (64, 3)).astype(float)
    k[~k.any(1)] = 1.0
    a = r.standard_normal((64, 3))
    a *= (np.linalg.norm(k, axis=1) ** -3 / np.linalg.norm(a, axis=1))[:, None]
    ph = r.uniform(0, 2 * np.pi, 64)
    x = np.stack(np.meshgrid(*[np.linspace(0, 1, 17)] * 3, indexing="ij"), -1).reshape(-1, 3)
    f, df = x * (1 - x), 1 - 2 * x
    B = 64 * f.prod(1, keepdims=True)
    dB = 64 * np.stack([df[:, c] * f[:, c - 1] * f[:, c - 2] for c in range(3)], 1)
    th = 2 * np.pi * x @ k.T + ph
    v = np.cross(2 * B * dB, np.sin(th) @ a) + B ** 2 * (np.cos(th) @ (2 * np.pi * np.cross(k, a)))
    return g.curl_modes(k, a, ph, 0.1 / np.linalg.norm(v, axis=1).max())


def padded(params):
    """The parameters as one flat array: every one starts at a multiple of four (gnn_layout)."""
    return torch.cat([torch.nn.functional.pad(w.reshape(-1), (0, -w.numel() % 4)) for w in params])


def weights(case, seed):
    """The network's parameters, in the order of gnn_layout: We, be, (Ws, Wm, b) per layer, Wd, bd."""
    C = (case["pt"] + 1) * len(multi_indices(case["p"]))
    gen = torch.Generator().manual_seed(seed)
    shapes = [(HIDDEN, C + 2), (HIDDEN,)] + [(HIDDEN, HIDDEN), (HIDDEN, HIDDEN), (HIDDEN,)] * LAYERS + [(C, HIDDEN), (C,)]
    return [torch.randn(*s, generator=gen) * (0.8 / math.sqrt(s[-1]) if len(s) == 2 else 0.1) for s in shapes]


def inputs(case, seed, ne, nf):
    """The device arrays of a case, by name."""
    gen = torch.Generator(device=DEV).manual_seed(seed)
    kind = case["kind"]
    if kind == "solve":
        b = smooth((ne,), case, gen)
        b[0, :, 0] = 0.0                          # the pinned rows
        return {"b": b.reshape(-1)}
    if kind == "apply":
        return {"x": smooth((ne,), case, gen).reshape(-1)}
    if kind == "apply_f32":
        return {"x": smooth((ne,), case, gen).float().reshape(-1)}
    if kind == "rhs":
        return {"F": smooth((nf, 3), case, gen).reshape(-1)}
    if kind == "update":
        return {"F": smooth((nf, 3), case, gen).reshape(-1), "dp": smooth((ne,), case, gen).reshape(-1)}
    if kind == "convection":
        return {"vbar": 0.1 * smooth((3, ne), case, gen).reshape(-1)}
    if kind == "gnn_grad":
        return {"R": smooth((case["pairs"], ne), case, gen).reshape(-1),
                "T": smooth((case["pairs"], ne), case, gen).reshape(-1)}
    if kind == "gnn_apply":
        return {"r": smooth((ne,), case, gen).reshape(-1)}
    return {}


def prepare(case, seed):
    mesh = g.Mesh(*kuhn_mesh(case["n"], seed))
    s = g.Solver(mesh, g.Reference(case["p"], case["pt"]), DT, precision=case["precision"])
    state = {"case": case, "solver": s, **inputs(case, seed, mesh.ne, mesh.nf)}
    kind = case["kind"]
    if kind == "step":
        if case["data"] == "solenoidal":
            s.set_initial(solenoidal(seed))
            s.set_boundary(g.zero())
        else:
            field = g.beltrami(np.pi / 4, np.pi / 2, case["nu"])
            s.set_initial(field)
            s.set_boundary(field)
        state["P"], state["V"], state["t"] = s.get_state()
    elif kind == "apply" or kind == "solve":
        state["y"] = s.pressure_empty()
    elif kind == "apply_f32":
        state["y"] = torch.empty_like(state["x"])
    elif kind == "rhs":
        state["b"] = s.pressure_empty()
    elif kind == "update":
        state["V"] = s.velocity_empty()
    elif kind == "convection":
        s.set_boundary(g.zero())
        state["ups"] = torch.empty_like(state["vbar"])
    elif kind.startswith("gnn"):
        s.gnn_init(hidden=HIDDEN, layers=LAYERS, bf16=case["bf16"], seed=0)
        s.gnn_params(padded(weights(case, seed)).numpy())
        state["z"] = s.pressure_empty()
    return state


def run(state):
    case, s, kind = state["case"], state["solver"], state["case"]["kind"]
    if kind == "step":
        s.set_state(state["P"], state["V"], state["t"])
        s.step(case["nu"], case["npic"], method=case["method"], tol=case["tol"])
        P, V, _ = s.get_state()
        return {"P": P, "V": V}
    if kind == "solve":
        return s.solve(state["b"], tol=case["tol"], method=case["method"], x=state["y"])[0]
    if kind == "apply":
        return s.pressure_apply(state["x"], state["y"])
    if kind == "apply_f32":
        return s.pressure_apply_f32(state["x"], state["y"])
    if kind == "rhs":
        return s.pressure_rhs(state["F"], state["b"])
    if kind == "update":
        return s.velocity_update(state["F"], state["dp"], state["V"])
    if kind == "convection":
        return s.convection(state["vbar"], state["ups"])
    if kind == "gnn_grad":
        loss, grad = s.gnn_loss_grad(state["R"], state["T"], case["pairs"])
        return {"loss": loss, "grad": grad}
    return s.gnn_apply(state["r"], state["z"])


# --------------------------------------------------------------------------------------------------- work
def work(case):
    n, p, Ng = case["n"], case["p"], case["pt"] + 1
    ne, nb = 6 * n ** 3, 12 * n * n
    nint = (4 * ne - nb) // 2
    nf, N = nint + nb, len(multi_indices(p))
    Nst, sides = N * Ng, 2 * nint + nb
    kind = case["kind"]
    entry = {"fp64": 8, "df32": 8, "mixed_f32": 4, "mixed_bf16": 2}[case["precision"]]
    vec = 4 if kind == "apply_f32" else 8
    entries = ne * N * (N + 1) // 2 + nint * N * N          # symmetric diagonal blocks, one block per face
    op = {"bytes": entry * entries + 2 * vec * ne * Nst, "flops": 2 * Ng * (ne * N * N + 2 * nint * N * N)}
    if kind.startswith("apply"):
        return op
    if kind == "rhs":
        return {"bytes": 8 * (3 * N * N * sides + 3 * nf * Nst + ne * Nst), "flops": 2 * 3 * N * Nst * sides}
    if kind == "update":
        return {"bytes": 8 * (6 * N * N * nint + 6 * nf * Nst + ne * Nst), "flops": 2 * 6 * N * Nst * nint}
    nq1 = math.ceil((3 * p + 2) / 2)
    conv = {"bytes": 8 * 6 * ne * Nst, "flops": 2 * ne * Nst * (12 * nq1 ** 3 + 4 * 9 * nq1 ** 2)}
    if kind == "convection":
        return conv
    if kind.startswith("gnn"):
        params = HIDDEN * (2 * Nst + 2) + 2 * LAYERS * HIDDEN ** 2
        passes, npair = (3, case["pairs"]) if kind == "gnn_grad" else (1, 1)
        return {"bytes": 8 * 2 * npair * ne * Nst, "flops": 2 * passes * npair * ne * params}
    # solves: 200 operator applications, about what the coarse-corrected iteration takes at every size
    its = {"bytes": 200 * op["bytes"], "flops": 200 * op["flops"]}
    if kind == "solve":
        return its
    # a Picard iteration: the pressure solve, three viscous solves of about 35 applications each, the
    # convection and six passes over the per-face blocks
    k = case["npic"]
    return {"bytes": k * (1.5 * its["bytes"] + conv["bytes"] + 8 * 18 * N * N * nf),
            "flops": k * (1.5 * its["flops"] + conv["flops"] + 2 * 18 * N * Nst * nf)}


# -------------------------------------------------------------------------------------------------- exact
def gauss_jacobi(n, alpha):
    """n-point rule on [0, 1] for the weight (1 - x)^alpha, by the recurrence's eigenvalues."""
    k = np.arange(n, dtype=float)
    s = 2 * k + alpha
    a = np.where(s * (s + 2) == 0, -alpha / (alpha + 2), -alpha ** 2 / np.where(s * (s + 2) == 0, 1, s * (s + 2)))
    k, s = k[1:], s[1:]
    b = np.sqrt(4 * k ** 2 * (k + alpha) ** 2 / (s ** 2 * (s + 1) * (s - 1)))
    x, v = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
    return (x + 1) / 2, v[0] ** 2 / (alpha + 1)


def collapsed_rule(n, dim):
    """Points (m, dim) and weights (m,) of the collapsed Gauss-Jacobi rule of the unit simplex."""
    rules = [gauss_jacobi(n, a) for a in range(dim)]
    g1 = np.meshgrid(*[r[0] for r in rules], indexing="ij")
    w = functools.reduce(np.multiply.outer, [r[1] for r in rules])
    pts = [functools.reduce(np.multiply, [1 - q for q in g1[c + 1:]], g1[c]) for c in range(dim)]
    t = lambda z: torch.as_tensor(np.ascontiguousarray(z), dtype=torch.float64, device=DEV)  # noqa: E731
    return t(np.stack([q.ravel() for q in pts], 1)), t(w.ravel())


def jacobi(n, a, x):
    """P_0 .. P_n of the Jacobi weight (a, 0) at x."""
    out = [torch.ones_like(x), ((a + 2) * x + a) / 2]
    for k in range(2, n + 1):
        s = 2 * k + a
        out.append(((s - 1) * (s * (s - 2) * x + a * a) * out[-1] - 2 * (k + a - 1) * (k - 1) * s * out[-2])
                   / (2 * k * (k + a) * (s - 2)))
    return out[:n + 1]


def dubiner(p, xi):
    """Orthonormal Dubiner values (m, N) and reference gradients (m, N, 3) at xi (m, 3)."""
    xi = xi.clone().requires_grad_(True)
    x, y, z = xi.unbind(1)
    s, t = 1 - y - z, 1 - z
    P = jacobi(p, 0, 2 * x / s - 1)
    cols = []
    for i, j, k in multi_indices(p):
        c = math.sqrt((2 * i + 1) * (2 * i + 2 * j + 2) * (2 * i + 2 * j + 2 * k + 3))
        cols.append(c * s ** i * P[i] * t ** j * jacobi(j, 2 * i + 1, 2 * y / t - 1)[j]
                    * jacobi(k, 2 * i + 2 * j + 2, 2 * z - 1)[k])
    grads = [torch.autograd.grad(c.sum(), xi, retain_graph=True)[0] for c in cols]
    return torch.stack(cols, 1).detach(), torch.stack(grads, 1).detach()


def legendre(pt, tau):
    """Orthonormal Legendre values and derivatives on [0, 1], (m, pt + 1)."""
    L = [np.polynomial.legendre.Legendre.basis(a, domain=[0, 1]) * math.sqrt(2 * a + 1) for a in range(pt + 1)]
    return np.stack([q(tau) for q in L], 1), np.stack([q.deriv()(tau) for q in L], 1)


class Scheme:
    """The discretisation of one case in binary64: geometry, face tables and the blocks Q."""

    def __init__(self, case, seed):
        self.p, self.pt = case["p"], case["pt"]
        self.N, self.Ng = len(multi_indices(self.p)), self.pt + 1
        verts, tets = kuhn_mesh(case["n"], seed)
        ne = self.ne = len(tets)
        # faces: local face f is opposite vertex f; left = lower tet; numbered by (left, local face)
        tri = np.stack([np.delete(tets, f, 1) for f in range(4)], 1)                  # (ne, 4, 3)
        key = np.sort(tri.reshape(-1, 3), 1)
        _, inv, cnt = np.unique(key, axis=0, return_inverse=True, return_counts=True)
        order = np.argsort(inv.ravel(), kind="stable")                                # the lower tet first
        first = np.cumsum(cnt) - cnt
        a = order[first]
        b = np.where(cnt == 2, order[np.minimum(first + 1, len(order) - 1)], -1)
        by = np.argsort(a)
        a, b = a[by], b[by]
        nf = self.nf = len(a)
        left, right = a // 4, np.where(b >= 0, b // 4, -1)
        fv = tri.reshape(-1, 3)[a]                                                    # left's local order
        where = lambda tet: (tets[tet][:, None, :] == fv[:, :, None]).argmax(2)       # noqa: E731
        code = lambda loc: loc[:, 0] * 16 + loc[:, 1] * 4 + loc[:, 2]                 # noqa: E731
        t = lambda v: torch.as_tensor(v, device=DEV)                                  # noqa: E731
        self.left, self.right = t(left), t(right)
        self.inner = self.right >= 0
        self.code = [t(code(where(left))), t(code(where(np.maximum(right, 0))))]
        X = t(verts)[t(tets)]                                                         # (ne, 4, 3)
        J = (X[:, 1:] - X[:, :1]).transpose(1, 2)
        self.det, self.Jinv, self.bary = torch.linalg.det(J), torch.linalg.inv(J), X.mean(1)
        self.fv = t(verts)[t(fv)]                                                     # (nf, 3, 3)
        cr = torch.linalg.cross(self.fv[:, 1] - self.fv[:, 0], self.fv[:, 2] - self.fv[:, 0])
        self.area2 = cr.norm(dim=1)
        away = self.fv[:, 0] - self.bary[self.left]
        self.normal = cr / self.area2[:, None] * torch.sign((cr * away).sum(1, keepdim=True))
        tau, w = gauss_jacobi(self.pt + 1, 0)
        v, d = legendre(self.pt, tau)
        v1 = legendre(self.pt, np.ones(1))[0][0]
        self.K = t(np.outer(v1, v1) - (d * w[:, None]).T @ v)

    def codes(self, pts, dim):
        """Values and gradients of the tet basis at the points of a sub-tet (dim 3) or face (dim 2) rule, for
        every code of the face's vertices in the tet."""
        V = torch.tensor([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1]], dtype=torch.float64, device=DEV)
        m = len(pts)
        val = torch.zeros(64, m, self.N, dtype=torch.float64, device=DEV)
        grd = torch.zeros(64, m, self.N, 3, dtype=torch.float64, device=DEV)
        for a, b, c in itertools.permutations(range(4), 3):
            F = [V[b] - V[a], V[c] - V[a], torch.full_like(V[a], 0.25) - V[a]][:dim]
            val[a * 16 + b * 4 + c], grd[a * 16 + b * 4 + c] = dubiner(self.p, V[a] + pts @ torch.stack(F))
        return val, grd

    def blocks(self):
        """Q[f][s][c][m][l] = int_{T_sf} psi_m d_c phi_l - sigma n_c int_face psi_m phi_l."""
        (sp, sw), (fp, fw) = collapsed_rule(self.p + 1, 3), collapsed_rule(self.p + 1, 2)
        sv, sg = self.codes(sp, 3)
        tv, _ = self.codes(fp, 2)
        N, ex = self.N, multi_indices(self.p)
        Q = torch.empty(self.nf, 2, 3, N, N, dtype=torch.float64, device=DEV)
        for at in torch.arange(self.nf, device=DEV).split(8192):
            F, tets = self.fv[at], [self.left[at], self.right[at].clamp(min=0)]
            ok = [torch.ones_like(self.area2[at]), self.inner[at].double()]
            E = [torch.stack([F[:, 1] - F[:, 0], F[:, 2] - F[:, 0], self.bary[i] - F[:, 0]], 1) for i in tets]
            x = [F[:, :1] + torch.einsum("qe,fed->fqd", sp, e) for e in E]
            w = [sw * (torch.linalg.det(e).abs() * o)[:, None] for e, o in zip(E, ok)]
            far = torch.cat([F, self.bary[tets[0]][:, None], torch.where(self.inner[at][:, None], self.bary[tets[1]],
                                                                          self.bary[tets[0]])[:, None]], 1)
            lo, hi = far.min(1).values, far.max(1).values
            # products of Legendre polynomials: the same flag as the Taylor monomials, so the same
            # Gram-Schmidt result, but well conditioned

            def taylor(q):
                y = (2 * q - (lo + hi)[:, None]) / (hi - lo)[:, None]
                L = [jacobi(max(self.p, 1), 0, y[..., d]) for d in range(3)]
                return torch.stack([L[0][i] * L[1][j] * L[2][k] for i, j, k in ex], -1)

            psi, face = [taylor(q) for q in x], taylor(F[:, :1] + torch.einsum("qe,fed->fqd", fp, torch.stack(
                [F[:, 1] - F[:, 0], F[:, 2] - F[:, 0]], 1)))
            for _ in range(2):                    # two Cholesky passes: orthonormal to rounding
                G = sum(torch.einsum("fqm,fq,fqn->fmn", a, b, a) for a, b in zip(psi, w))
                R = torch.linalg.cholesky(G)
                solve = lambda z: torch.linalg.solve_triangular(R, z.transpose(1, 2), upper=False).transpose(1, 2)  # noqa: E731
                psi, face = [solve(a) for a in psi], solve(face)
            for s in range(2):
                c = self.code[s][at]
                vol = torch.einsum("fqm,fqle,fed->fdml", psi[s] * w[s][..., None], sg[c], self.Jinv[tets[s]])
                bd = torch.einsum("fqm,q,fql->fml", face, fw, tv[c]) * (self.area2[at] * ok[s])[:, None, None]
                sig = 1.0 if s == 0 else -1.0
                Q[at, s] = vol - sig * self.normal[at][:, :, None, None] * bd[:, None]
        return Q

    def gradient(self, Q, x):
        """Sum_s Q_s x_s per interior face, (f, 3, Ng, N); x (ne, Ng, N)."""
        f = self.inner.nonzero()[:, 0]
        return torch.einsum("fcml,fal->fcam", Q[f, 0], x[self.left[f]]) + \
            torch.einsum("fcml,fal->fcam", Q[f, 1], x[self.right[f]])

    def divergence(self, Q, F, faces):
        """- Sum_f Q_sf^T F_f per tet, (ne, Ng, N); F (len(faces), 3, Ng, N)."""
        y = torch.zeros(self.ne, self.Ng, self.N, dtype=torch.float64, device=DEV)
        y.index_add_(0, self.left[faces], torch.einsum("fcml,fcam->fal", Q[faces, 0], F), alpha=-1)
        in2 = self.inner[faces]
        f2 = faces[in2]
        y.index_add_(0, self.right[f2], torch.einsum("fcml,fcam->fal", Q[f2, 1], F[in2]), alpha=-1)
        return y

    def spatial(self, Q, x):
        """The spatial operator A_sp x with the pinned constant mode of tet 0 left out."""
        x = x.clone()
        x[0, :, 0] = 0
        y = self.divergence(Q, self.gradient(Q, x), self.inner.nonzero()[:, 0])
        y[0, :, 0] = 0
        return y


def exact_solve(S, Q, b):
    """A x = b by block-Jacobi conjugate gradients on the columns of A_sp X = K b / dt^2, to rounding."""
    rhs = -torch.einsum("ab,ibk->iak", S.K, b) / DT ** 2
    f = S.inner.nonzero()[:, 0]
    D = torch.zeros(S.ne, S.N, S.N, dtype=torch.float64, device=DEV)
    for s, side in ((0, S.left), (1, S.right)):
        D.index_add_(0, side[f], torch.einsum("fcml,fcmk->flk", Q[f, s], Q[f, s]))
    D[0, 0, :] = 0
    D[0, :, 0] = 0
    D[0, 0, 0] = 1
    Dinv = torch.linalg.inv(D)
    pre = lambda r: torch.einsum("ikl,ial->iak", Dinv, r)                              # noqa: E731
    dot = lambda u, v: (u * v).sum((0, 2))                                             # noqa: E731
    x, r = torch.zeros_like(rhs), rhs.clone()
    z = pre(r)
    p, rz, goal = z.clone(), dot(r, z), 1e-15 * rhs.norm()
    for it in range(3000):
        q = -S.spatial(Q, p)
        al = rz / dot(p, q).clamp(min=1e-300)
        x += al[None, :, None] * p
        r -= al[None, :, None] * q
        if it % 20 == 0 and r.norm() <= goal:
            break
        z = pre(r)
        new = dot(r, z)
        p = z + (new / rz.clamp(min=1e-300))[None, :, None] * p
        rz = new
    return x


def exact_convection(S, vbar):
    """Ups of the Rusanov space-time DG convection on one slab, zero velocity beyond the walls."""
    nq = math.ceil((3 * S.p + 2) / 2)
    (vp, vw), (fp, fw) = collapsed_rule(nq, 3), collapsed_rule(nq, 2)
    tau, tw = gauss_jacobi(math.ceil((3 * S.pt + 2) / 2), 0)
    gam = torch.as_tensor(legendre(S.pt, tau)[0], device=DEV)
    tw = torch.as_tensor(tw, device=DEV)
    val, grd = dubiner(S.p, vp)
    fval, _ = S.codes(fp, 2)
    V = vbar.reshape(3, S.ne, S.Ng, S.N).transpose(0, 1)                               # (ne, 3, Ng, N)
    out = torch.zeros_like(V)
    for at in torch.arange(S.ne, device=DEV).split(2048):
        v = torch.einsum("icbk,qk,tb->icqt", V[at], val, gam)
        u = torch.einsum("ied,idqt->ieqt", S.Jinv[at], v)
        w = DT * S.det[at][:, None, None] * vw[:, None] * tw
        h = torch.einsum("iqt,icqt,ieqt,ta->iceqa", w, v, u, gam)
        out[at] -= torch.einsum("iceqa,qke->icak", h, grd)
    for at in torch.arange(S.nf, device=DEV).split(4096):
        l, r = S.left[at], S.right[at].clamp(min=0)
        cl, cr = fval[S.code[0][at]], fval[S.code[1][at]]
        vm = torch.einsum("fcbk,fqk,tb->fcqt", V[l], cl, gam)
        vr = torch.einsum("fcbk,fqk,tb->fcqt", V[r], cr, gam) * S.inner[at][:, None, None, None]
        n = S.normal[at]
        flux = lambda q: q * torch.einsum("fdqt,fd->fqt", q, n)[:, None]               # noqa: E731
        smax = 2 * torch.maximum(vm.norm(dim=1), vr.norm(dim=1))[:, None]
        H = 0.5 * (flux(vm) + flux(vr)) - 0.5 * smax * (vr - vm)
        H = H * (DT * S.area2[at][:, None, None] * fw[:, None] * tw)[:, None]
        H = torch.einsum("fcqt,ta->fcqa", H, gam)
        out.index_add_(0, l, torch.einsum("fcqa,fqk->fcak", H, cl))
        i2 = S.inner[at]
        out.index_add_(0, r[i2], torch.einsum("fcqa,fqk->fcak", H[i2], cr[i2]), alpha=-1)
    return out.transpose(0, 1).reshape(-1)


def exact_network(S, case, seed, data):
    params = [w.to(DEV).double().requires_grad_(True) for w in weights(case, seed)]
    nbr = torch.full((S.ne, 4), -1, dtype=torch.int64, device=DEV)
    f = S.inner.nonzero()[:, 0]
    ends = torch.cat([torch.stack([S.left[f], S.right[f]], 1), torch.stack([S.right[f], S.left[f]], 1)])
    walls = torch.zeros(S.ne, dtype=torch.float64, device=DEV).index_add_(
        0, S.left[~S.inner], torch.ones(int((~S.inner).sum()), dtype=torch.float64, device=DEV))
    geom = torch.stack([(S.det / S.det.mean()) ** (1 / 3), walls / 4], 1)

    def net(r):
        r = r.reshape(S.ne, -1)
        s = r.square().mean().sqrt()
        We, be, *mid, Wd, bd = params
        h = torch.relu(torch.cat([r / s, geom], 1) @ We.T + be)
        for k in range(LAYERS):
            Ws, Wm, b = mid[3 * k:3 * k + 3]
            m = torch.zeros_like(h).index_add(0, ends[:, 0], h[ends[:, 1]])
            h = torch.relu(h @ Ws.T + m @ Wm.T + b)
        return s * (h @ Wd.T + bd)

    if case["kind"] == "gnn_apply":
        return net(data["r"]).detach().reshape(-1)
    loss = 0.0
    for r, t in zip(data["R"].chunk(case["pairs"]), data["T"].chunk(case["pairs"])):
        loss = loss + (net(r) - t.reshape(S.ne, -1)).square().sum() / t.square().sum() / case["pairs"]
    grads = torch.autograd.grad(loss, params)
    return {"loss": float(loss), "grad": padded(grads).cpu().numpy()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "step":
        return None                               # a whole step in plain torch takes minutes
    S = Scheme(case, seed)
    data = inputs(case, seed, S.ne, S.nf)
    if kind.startswith("gnn"):
        return exact_network(S, case, seed, data)
    if kind == "convection":
        return exact_convection(S, data["vbar"])
    Q = S.blocks()
    shape = (S.ne, S.Ng, S.N)
    if kind == "solve":
        return exact_solve(S, Q, data["b"].reshape(shape)).reshape(-1)
    if kind == "rhs":
        b = DT * S.divergence(Q, data["F"].reshape(S.nf, 3, S.Ng, S.N), torch.arange(S.nf, device=DEV))
        b[0, :, 0] = 0
        return b.reshape(-1)
    Kinv = torch.linalg.inv(S.K)
    if kind == "update":
        V = data["F"].reshape(S.nf, 3, S.Ng, S.N).clone()
        V[S.inner] -= DT * torch.einsum("ab,fcbm->fcam", Kinv, S.gradient(Q, data["dp"].reshape(shape)))
        return V.reshape(-1)
    x = data["x"].double().reshape(shape)
    y = DT ** 2 * torch.einsum("ab,ibk->iak", Kinv, S.spatial(Q, x))
    y[0, :, 0] = -x[0, :, 0]
    return y.reshape(-1)
