"""stdg_profile_read's kernel_launches is the number of kernels that ran, as the CUDA profiler of PyTorch sees them."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from inputs import kuhn_mesh


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1601_07384_gb300.build import build
    build()


def ran(call):
    """Kernels of one call (copies and memsets apart); PyTorch itself launches none in these calls."""
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        call()
        torch.cuda.synchronize()
    return sum(e.device_type.name == "CUDA" and not e.name.startswith("Mem") for e in prof.events())


@pytest.mark.parametrize("precision,graph_batch", [("fp64", 8), ("fp64", 1), ("df32", 8), ("mixed_f32", 8), ("mixed_f32", 1)])
@pytest.mark.parametrize("p,pt", [(1, 0), (2, 1)])
def test_launches_are_counted(precision, graph_batch, p, pt):
    import paper_1601_07384_gb300 as g
    s = g.Solver(g.Mesh(*kuhn_mesh(3, seed=0)), g.Reference(p, pt), 0.01, precision=precision, graph_batch=graph_batch)
    field = g.beltrami(1.0, 1.0, 0.1)
    s.set_boundary(field)
    s.set_initial(field)
    P, V, t = s.get_state()
    gen = torch.Generator().manual_seed(1)
    x, b, F, vbar = (torch.randn(n, generator=gen, dtype=torch.float64).cuda()
                     for n in (P.numel(), P.numel(), V.numel(), 3 * P.numel()))
    b.view(s.ne, s.Ng, s.N)[0, :, 0] = 0.0
    y, U, W, ups = torch.empty_like(x), torch.empty(2 * V.numel(), dtype=torch.float64, device="cuda"), \
        torch.empty_like(V), torch.empty_like(vbar)

    def step():
        s.set_state(P, V, t)
        s.step(0.1, 2, method="kron_mg", tol=1e-9)

    calls = {"apply": lambda: s.pressure_apply(x, y), "factored": lambda: s.pressure_apply_factored(x, y),
             "rhs": lambda: s.pressure_rhs(F, y), "update": lambda: s.velocity_update(F, x, W),
             "moments": lambda: s.velocity_moments(F, U), "convection": lambda: s.convection(vbar, ups), "step": step}
    for method in ("kron_cg", "kron_pcg", "kron_mg"):
        calls[method] = lambda method=method: s.solve(b, tol=1e-9, method=method, x=y)
    if precision == "fp64":
        calls["gmres"] = lambda: s.solve(b, tol=1e-6, method="gmres", x=y)
    ran(lambda: s.pressure_apply(x, y))                       # the profiler's own start
    for name, call in calls.items():
        call()                                                # first calls build tables and arrays
        want = ran(call)
        s.profile(False)
        call()
        assert s.profile_read()["kernel_launches"] == want, name
