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
