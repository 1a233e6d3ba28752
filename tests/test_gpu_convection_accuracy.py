"""The convective term's rounding error and its first call.

The rounding error against the binary64 oracle: the kernels with the degrees at compile time
are at least as accurate as the general kernel (STDG_CONV_KERNEL=generic), which sums every test function over the
points themselves, at every degree."""
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from inputs import kuhn_mesh
from oracle import operators as ops
from oracle.basis import multi_indices
from oracle.blocks import SpaceTimeDG
from oracle.mesh import Mesh


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1601_07384_gb300.build import build
    build()


@pytest.mark.parametrize("p,pt", [(p, pt) for p in (1, 2, 3, 4) for pt in range(5)])
@pytest.mark.parametrize("data", ["resolved", "random"])
def test_rounding_error_is_no_larger_than_the_general_kernels(p, pt, data, monkeypatch):
    """Root mean square over a few thousand outputs (one or two per cent of noise)."""
    import paper_1601_07384_gb300 as g
    n = {1: 4, 2: 3, 3: 2, 4: 2}[p]
    d = SpaceTimeDG(Mesh(*kuhn_mesh(n, seed=0)), p, pt, 0.01)
    rng, err = np.random.default_rng(10 * p + pt), {"default": 0.0, "generic": 0.0}
    fall = 1.0
    if data == "resolved":
        deg = np.array([sum(e) for e in multi_indices(p)])
        fall = (0.3 ** np.arange(pt + 1)[:, None] * 0.5 ** deg[None, :]).ravel()
    for _ in range(2):
        vbar = rng.standard_normal((d.mesh.ne, 3, d.Nst)) * fall
        exact = ops.convection(d, vbar, 0.0, lambda x, t: np.zeros((len(x), 3)))
        for kernel in err:
            if kernel == "generic":
                monkeypatch.setenv("STDG_CONV_KERNEL", "generic")
            else:
                monkeypatch.delenv("STDG_CONV_KERNEL", raising=False)
            s = g.Solver(g.Mesh(*kuhn_mesh(n, seed=0)), g.Reference(p, pt), 0.01)
            s.set_boundary(g.zero())
            out = s.convection(torch.from_numpy(np.ascontiguousarray(vbar.transpose(1, 0, 2))).cuda())
            out = out.cpu().numpy().reshape(3, d.mesh.ne, d.Nst).transpose(1, 0, 2)
            err[kernel] += np.square(out - exact).sum() / np.square(exact).sum()
    print(f"p={p} pt={pt} {data}: rms error {np.sqrt(err['default'] / 2):.2e}, general {np.sqrt(err['generic'] / 2):.2e}")
    assert err["default"] <= err["generic"]


@pytest.mark.parametrize("p,pt", [(3, 1), (4, 4)])
def test_first_call_of_a_solver_builds_its_tables_quickly(p, pt):
    """The tables of the degrees are built in the first call, on the device: medians over five solvers, with room for
    six later calls and half a millisecond (evaluated on the host they took 0.9 and 2.5 ms)."""
    import paper_1601_07384_gb300 as g
    first, later = [], []
    for k in range(6):
        s = g.Solver(g.Mesh(*kuhn_mesh(2, seed=k)), g.Reference(p, pt), 0.01)
        s.set_boundary(g.zero())
        vbar = torch.ones(3 * s.ne * s.Nst, dtype=torch.float64, device="cuda")
        ups = torch.empty_like(vbar)
        for out in (first, later):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            s.convection(vbar, ups)
            torch.cuda.synchronize()
            out.append(time.perf_counter() - t0)
    f, l = np.median(first[1:]), np.median(later[1:])
    print(f"p={p} pt={pt}: first {f * 1e6:.0f} us, later {l * 1e6:.0f} us")
    assert f <= 6 * l + 5e-4
