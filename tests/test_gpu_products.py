"""The block products, vector reductions and the convection over all compiled degrees, 0 <= p, p_t <= 4: every
(N, Ng) is an instantiation of its own with its own split of rows, columns and units over the threads.

Tolerances: a product or the convective term agrees to 1e-12 of the largest output, as everywhere in
test_gpu_parity.py; solves are judged by their residual with the oracle's operator."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from inputs import BeltramiParams, beltrami_velocity, kuhn_mesh
from oracle import operators as ops
from oracle.blocks import SpaceTimeDG
from oracle.mesh import Mesh
from oracle.step import initial_state, time_step

DEGREES = [(p, pt) for p in range(5) for pt in range(5)]


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1601_07384_gb300.build import build
    build()


def setup(n, p, pt, dt=0.01, **kw):
    import paper_1601_07384_gb300 as g
    v, t = kuhn_mesh(n, seed=0)
    return g.Solver(g.Mesh(v, t), g.Reference(p, pt), dt, **kw), SpaceTimeDG(Mesh(v, t), p, pt, dt)


def rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / max(np.abs(np.asarray(b)).max(), 1e-300)


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("p,pt", DEGREES)
def test_products_match_oracle_at_every_degree(p, pt):
    """Five-point operator (pinned and not), its factored form, velocity update and right-hand side."""
    gs, d = setup(2, p, pt)
    m, rng = d.mesh, np.random.default_rng(10 * p + pt)
    x, F = rng.standard_normal((m.ne, d.Nst)), np.zeros((m.nf, 3, d.Nst))
    for pinned in (True, False):
        yo = ops.pressure_apply(d, x, pinned=pinned).ravel()
        assert rel(gs.pressure_apply(cuda(x.ravel()), pinned=pinned).cpu().numpy(), yo) <= 1e-12
        assert rel(gs.pressure_apply_factored(cuda(x.ravel()), pinned=pinned).cpu().numpy(), yo) <= 1e-12
    V = gs.velocity_update(cuda(F.ravel()), cuda(x.ravel()))
    U = gs.velocity_moments(V).cpu().numpy().reshape(m.nf, 2, 3, d.Nst)
    Vo = ops.velocity_update(d, F, x, np.zeros((m.nf, 3, d.Nst)))
    Uo = np.zeros_like(U)
    for j in range(m.nf):
        fb = d.face_blocks(j)
        for s in range(len(fb["sides"])):
            Uo[j, s] = (fb["Mij"][s] @ Vo[j].T).T
    assert rel(U, Uo) <= 1e-12
    assert rel(gs.pressure_rhs(V, pinned=False).cpu().numpy(), ops.pressure_rhs(d, Vo, pinned=False).ravel()) <= 1e-11


@pytest.mark.parametrize("p,pt", [(0, 2), (1, 0), (1, 4), (2, 1), (3, 3), (4, 0)])
def test_products_with_unequal_scales(p, pt):
    """Tets whose values lie hundreds of orders of magnitude apart, down to the subnormal range: each
    output tet is as accurate as the largest of the tets that it reads allows."""
    gs, d = setup(2, p, pt)
    m, rng = d.mesh, np.random.default_rng(3)
    x = rng.standard_normal((m.ne, d.Nst))
    size = 10.0 ** rng.choice([-315.0, -300.0, -150.0, 0.0, 120.0], m.ne)
    x *= size[:, None]
    y = gs.pressure_apply(cuda(x.ravel()), pinned=False).cpu().numpy().reshape(m.ne, d.Nst)
    yo = ops.pressure_apply(d, x, pinned=False).reshape(m.ne, d.Nst)
    unit = np.abs(ops.pressure_apply(d, rng.standard_normal((m.ne, d.Nst)), pinned=False)).max()
    most = np.abs(x).max(1)
    reach = most.copy()
    for j in np.nonzero(m.interior)[0]:
        l, r = m.left[j], m.right[j]
        reach[l], reach[r] = max(reach[l], most[r]), max(reach[r], most[l])
    assert (np.abs(y - yo).max(1) <= 1e-12 * unit * reach + 1e-320).all()


@pytest.mark.parametrize("p,pt", [(0, 2), (1, 4), (2, 1), (3, 0), (4, 4)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_products_carry_non_finite_values(p, pt, bad):
    """A non-finite value reaches its tet and the neighbours across the faces, and nothing else."""
    gs, d = setup(2, p, pt)
    m = d.mesh
    x = np.random.default_rng(4).standard_normal((m.ne, d.Nst))
    clean = gs.pressure_apply(cuda(x.ravel()), pinned=False).cpu().numpy().reshape(m.ne, d.Nst)
    x[m.ne // 2, d.Nst - 1] = bad
    y = gs.pressure_apply(cuda(x.ravel()), pinned=False).cpu().numpy().reshape(m.ne, d.Nst)
    near = {m.ne // 2}
    for j in np.nonzero(m.interior)[0]:
        if m.ne // 2 in (m.left[j], m.right[j]):
            near |= {m.left[j], m.right[j]}
    hit = np.isin(np.arange(m.ne), list(near))
    assert not np.isfinite(y[hit]).all(1).any()
    # other tets: as before, up to the rounding of another path for a unit that shares a CTA
    assert rel(y[~hit], clean[~hit]) <= 1e-14


@pytest.mark.parametrize("p,pt", [(p, pt) for p, pt in DEGREES if p > 0])
def test_solves_reach_their_tolerance_at_every_degree(p, pt):
    """The decoupled solvers in binary64 and with binary32 inner iterations, true residual by the oracle."""
    d = None
    for precision, method in (("fp64", "kron_cg"), ("fp64", "kron_pcg"), ("mixed_f32", "kron_pcg"), ("mixed_f32", "kron_mg")):
        if d is None:
            gs, d = setup(2, p, pt, precision=precision)
            b = np.random.default_rng(8).standard_normal((d.mesh.ne, d.Nst))
            b[0, ops.pin_index(d)] = 0.0
        else:
            import paper_1601_07384_gb300 as g
            gs = g.Solver(g.Mesh(*kuhn_mesh(2, seed=0)), g.Reference(p, pt), 0.01, precision=precision)
        x, st = gs.solve(cuda(b.ravel()), tol=1e-11, method=method)
        r = b - ops.pressure_apply(d, x.cpu().numpy()).reshape(b.shape)
        assert np.linalg.norm(r) <= 1e-10 * np.linalg.norm(b), (precision, method, st)


@pytest.mark.parametrize("p,pt", [(p, pt) for p, pt in DEGREES if p > 0])
@pytest.mark.parametrize("data", ["beltrami", "zero"])
def test_convection_matches_general_kernel_at_every_degree(p, pt, data, monkeypatch):
    """The kernels with the degrees at compile time against the general one, values of order 1 in every
    mode (no decay that would hide an error in the high modes)."""
    import paper_1601_07384_gb300 as g
    prm, out = BeltramiParams(nu=0.1), []
    for kernel in ("default", "generic"):
        if kernel == "generic":
            monkeypatch.setenv("STDG_CONV_KERNEL", "generic")
        gs = g.Solver(g.Mesh(*kuhn_mesh(2, seed=0)), g.Reference(p, pt), 0.01)
        gs.set_boundary(g.beltrami(prm.a, prm.d, prm.nu) if data == "beltrami" else g.zero())
        vbar = np.random.default_rng(17).standard_normal(3 * gs.pressure_empty().numel())
        out.append(gs.convection(cuda(vbar)).cpu().numpy().ravel())
    assert rel(out[0], out[1]) <= 1e-12


@pytest.mark.parametrize("p,pt", [(1, 4), (2, 3), (3, 2)])
def test_step_matches_oracle_at_other_degrees(p, pt):
    """Averaging, face gradient and go back within a Picard step, Beltrami data."""
    import paper_1601_07384_gb300 as g
    prm = BeltramiParams(nu=0.1)
    gs, d = setup(2, p, pt)
    field = g.beltrami(prm.a, prm.d, prm.nu)
    gs.set_initial(field)
    gs.set_boundary(field)
    gs.step(prm.nu, 2, method="kron_cg", tol=1e-13)
    P, V, _ = gs.get_state()
    so = initial_state(d, lambda x: beltrami_velocity(x, 0.0, prm))
    so = time_step(d, so, prm.nu, 2, lambda x, tt: beltrami_velocity(x, tt, prm), tol=1e-13, method="direct")
    U = gs.velocity_moments(V).cpu().numpy().reshape(d.mesh.nf, 2, 3, d.Nst)
    Uo = np.zeros_like(U)
    for j in range(d.mesh.nf):
        fb = d.face_blocks(j)
        for s in range(len(fb["sides"])):
            Uo[j, s] = (fb["Mij"][s] @ so.V[j].T).T
    assert rel(P.cpu().numpy(), so.P.ravel()) <= 1e-10
    assert rel(U, Uo) <= 1e-10


@pytest.mark.parametrize("pt", range(5))
@pytest.mark.parametrize("precision,tol", [("mixed_f32", 4e-6), ("mixed_bf16", 2e-2)])
@pytest.mark.parametrize("n", [2, 5, 9, 10])
def test_low_precision_operator_at_p4(n, pt, precision, tol):
    """Five warps per tet: fewer tets than CTAs, a few per CTA (both stages reused), and sizes on either side of
    the line above which bfloat16 blocks take the kernel with one warp per tet; against the binary64 product."""
    import paper_1601_07384_gb300 as g
    gs = g.Solver(g.Mesh(*kuhn_mesh(n, seed=0)), g.Reference(4, pt), 0.01, precision=precision)
    x = torch.randn(gs.pressure_empty().numel(), generator=torch.Generator().manual_seed(n), dtype=torch.float32).cuda()
    for pinned in (True, False):
        y = gs.pressure_apply_f32(x, pinned=pinned).double()
        yo = gs.pressure_apply(x.double(), pinned=pinned)
        # the pinned row carries its own large diagonal entry: compare it apart
        sel = torch.ones_like(yo, dtype=torch.bool)
        if pinned:
            sel.view(-1)[torch.arange(pt + 1, device="cuda") * 35] = False
        assert float((y - yo)[sel].abs().max() / yo[sel].abs().max()) <= tol
