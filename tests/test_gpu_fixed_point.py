"""The products in 64-bit fixed point where their operands are unlike those of a regular mesh and resolved fields.

Tolerances: 1e-12 of the largest output, as everywhere in test_gpu_parity.py, taken for every part of the result
that the products form on its own (a component, a tet)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from inputs import kuhn_mesh
from oracle import operators as ops
from oracle.blocks import SpaceTimeDG
from oracle.mesh import Mesh


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1601_07384_gb300.build import build
    build()


def setup(n, p, pt, dt=0.01, stretch=(1.0, 1.0, 1.0)):
    import paper_1601_07384_gb300 as g
    v, t = kuhn_mesh(n, seed=0)
    v = v * np.array(stretch)
    return g.Solver(g.Mesh(v, t), g.Reference(p, pt), dt), SpaceTimeDG(Mesh(v, t), p, pt, dt)


def rel(a, b):
    return np.abs(np.asarray(a) - np.asarray(b)).max() / max(np.abs(np.asarray(b)).max(), 1e-300)


def cuda(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


@pytest.mark.parametrize("p,pt", [(1, 0), (1, 1), (2, 0)])
@pytest.mark.parametrize("axis", [0, 2])
def test_components_of_a_stretched_mesh_keep_their_accuracy(p, pt, axis):
    """A layer 2^-26 as thick as it is wide: Q of the two other components is smaller by that factor, and so is
    what it contributes.  Every component of F by itself in the right-hand side, every component of the update."""
    stretch = [1.0, 1.0, 1.0]
    stretch[axis] = 2.0 ** -26
    gs, d = setup(2, p, pt, stretch=stretch)
    m, rng = d.mesh, np.random.default_rng(5)
    for c in range(3):
        F = np.zeros((m.nf, 3, d.Nst))
        F[:, c] = rng.standard_normal((m.nf, d.Nst))
        b = gs.pressure_rhs(cuda(F.ravel()), pinned=False).cpu().numpy()
        assert rel(b, ops.pressure_rhs(d, F, pinned=False).ravel()) <= 1e-12, c
    x = rng.standard_normal((m.ne, d.Nst))
    V = gs.velocity_update(cuda(np.zeros(m.nf * 3 * d.Nst)), cuda(x.ravel()))
    U = gs.velocity_moments(V).cpu().numpy().reshape(m.nf, 2, 3, d.Nst)
    Vo = ops.velocity_update(d, np.zeros((m.nf, 3, d.Nst)), x, np.zeros((m.nf, 3, d.Nst)))
    Uo = np.zeros_like(U)
    for j in range(m.nf):
        fb = d.face_blocks(j)
        for s in range(len(fb["sides"])):
            Uo[j, s] = (fb["Mij"][s] @ Vo[j].T).T
    for c in range(3):
        assert rel(U[:, :, c], Uo[:, :, c]) <= 1e-12, c


@pytest.mark.parametrize("p,pt", [(p, pt) for p in range(5) for pt in range(5)])
def test_velocity_moments_match_oracle_at_every_degree(p, pt):
    """Velocities of order 1 on all faces, the boundary's with one side only."""
    gs, d = setup(2, p, pt)
    m = d.mesh
    V = np.random.default_rng(10 * p + pt).standard_normal((m.nf, 3, d.Nst))
    U = gs.velocity_moments(cuda(V.ravel())).cpu().numpy().reshape(m.nf, 2, 3, d.Nst)
    for j in range(m.nf):
        fb = d.face_blocks(j)
        for s, Mij in enumerate(fb["Mij"]):
            assert rel(U[j, s], (Mij @ V[j].T).T) <= 1e-12
        if len(fb["Mij"]) == 1:
            assert not U[j, 1].any()


DEGREES = [(p, pt) for p in range(5) for pt in range(5)]
SIZES = [-315.0, -300.0, -150.0, 0.0, 120.0]


@pytest.mark.parametrize("p,pt", DEGREES)
def test_update_and_right_hand_side_match_oracle_at_every_degree(p, pt):
    """Velocities of order 1 on all faces: the update's copy of the boundary faces and its sum with the input, the
    boundary faces' part of the right-hand side."""
    gs, d = setup(2, p, pt)
    m, rng = d.mesh, np.random.default_rng(10 * p + pt)
    x, F = rng.standard_normal((m.ne, d.Nst)), rng.standard_normal((m.nf, 3, d.Nst))
    Vo = ops.velocity_update(d, F, x, F)
    for out in (None, "in place"):
        Ft = cuda(F.ravel())
        V = gs.velocity_update(Ft, cuda(x.ravel()), Ft if out else None).cpu().numpy().reshape(F.shape)
        assert rel(V, Vo) <= 1e-12
        assert np.array_equal(V[~m.interior], F[~m.interior])
    for pinned in (True, False):
        b = gs.pressure_rhs(cuda(F.ravel()), pinned=pinned).cpu().numpy()
        assert rel(b, ops.pressure_rhs(d, F, pinned=pinned).ravel()) <= 1e-12


@pytest.mark.parametrize("p,pt", [(0, 2), (1, 0), (1, 4), (2, 1), (3, 3), (4, 0)])
def test_update_and_right_hand_side_with_unequal_scales(p, pt):
    """Faces and tets whose values lie hundreds of orders of magnitude apart, down to the subnormal range, where the
    products fall back to binary64 multiply-adds: each output as accurate as the largest of its inputs allows."""
    gs, d = setup(2, p, pt)
    m, rng = d.mesh, np.random.default_rng(3)
    F = rng.standard_normal((m.nf, 3, d.Nst))
    unit = np.abs(ops.pressure_rhs(d, F, pinned=False)).max()
    F *= 10.0 ** rng.choice(SIZES, m.nf)[:, None, None]
    b = gs.pressure_rhs(cuda(F.ravel()), pinned=False).cpu().numpy().reshape(m.ne, d.Nst)
    bo = ops.pressure_rhs(d, F, pinned=False)
    most, reach = np.abs(F).max((1, 2)), np.zeros(m.ne)
    for j in range(m.nf):
        for i in d.face_blocks(j)["sides"]:
            reach[i] = max(reach[i], most[j])
    assert (np.abs(b - bo).max(1) <= 1e-12 * unit * reach + 1e-320).all()
    x = rng.standard_normal((m.ne, d.Nst))
    unit = np.abs(ops.velocity_update(d, np.zeros_like(F), x, np.zeros_like(F))).max()
    x *= 10.0 ** rng.choice(SIZES, m.ne)[:, None]
    V = gs.velocity_update(cuda(F.ravel()), cuda(x.ravel())).cpu().numpy().reshape(F.shape)
    Vo = ops.velocity_update(d, F, x, F)
    size = np.abs(x).max(1)
    for j in range(m.nf):
        top = max(size[i] for i in d.face_blocks(j)["sides"]) if m.interior[j] else 0.0
        assert np.abs(V[j] - Vo[j]).max() <= 1e-12 * (unit * top + most[j]) + 1e-320, j


@pytest.mark.parametrize("p,pt", [(0, 2), (1, 4), (2, 1), (3, 0), (4, 4)])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_update_and_right_hand_side_carry_non_finite_values(p, pt, bad):
    """A non-finite value of a face reaches its tets, one of a tet its inner faces, and nothing else."""
    gs, d = setup(2, p, pt)
    m, rng = d.mesh, np.random.default_rng(4)
    x, F = rng.standard_normal((m.ne, d.Nst)), rng.standard_normal((m.nf, 3, d.Nst))
    rhs = lambda F: gs.pressure_rhs(cuda(F.ravel()), pinned=False).cpu().numpy().reshape(m.ne, d.Nst)   # noqa: E731
    upd = lambda x: gs.velocity_update(cuda(F.ravel()), cuda(x.ravel())).cpu().numpy().reshape(F.shape)  # noqa: E731
    clean, cleanV = rhs(F), upd(x)
    j = int(np.nonzero(m.interior)[0][3])
    Fb = F.copy()
    Fb[j, 1, d.Nst - 1] = bad
    b = rhs(Fb)
    hit = np.isin(np.arange(m.ne), [m.left[j], m.right[j]])
    assert not np.isfinite(b[hit]).all(1).any()
    assert rel(b[~hit], clean[~hit]) <= 1e-14       # up to the rounding of another path for a unit that shares a CTA
    i = m.ne // 2
    xb = x.copy()
    xb[i, d.Nst - 1] = bad
    V = upd(xb)
    hit = m.interior & ((m.left == i) | (m.right == i))
    assert not np.isfinite(V[hit]).all((1, 2)).any()
    assert rel(V[~hit], cleanV[~hit]) <= 1e-14


@pytest.mark.parametrize("p,pt", [(1, 0), (2, 1), (1, 3)])
def test_averaging_and_go_back_with_tiny_values_beside_ordinary_ones(p, pt):
    """A step from a state whose faces hold values of order 1 or of order 1e-305 (which the products form with binary64
    multiply-adds) against the oracle's."""
    import paper_1601_07384_gb300 as g
    from oracle.step import State, time_step
    gs, d = setup(2, p, pt)
    m, rng = d.mesh, np.random.default_rng(6)
    V = 0.1 * rng.standard_normal((m.nf, 3, d.Nst)) * np.where(rng.random(m.nf) < 0.5, 1.0, 1e-305)[:, None, None]
    gs.set_boundary(g.zero())
    gs.set_state(cuda(np.zeros(m.ne * d.Nst)), cuda(V.ravel()), 0.0)
    gs.step(0.1, 1, method="kron_cg", tol=1e-13)
    P, Vn, _ = gs.get_state()
    so = time_step(d, State(V=V, P=np.zeros((m.ne, d.Nst))), 0.1, 1, lambda x, t: np.zeros((len(x), 3)), tol=1e-13,
                   method="direct")
    assert rel(P.cpu().numpy(), so.P.ravel()) <= 1e-10
    assert rel(Vn.cpu().numpy(), so.V.ravel()) <= 1e-10
