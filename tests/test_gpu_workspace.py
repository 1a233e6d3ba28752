"""Device arrays are written only inside their bounds: every array of a solver gets a guard behind it, which must
come through a solve unchanged."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from inputs import kuhn_mesh

GUARD = 256 * 1024          # bytes behind every array


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1601_07384_gb300.build import build
    build()


@pytest.fixture
def guarded(monkeypatch):
    """The solver's arrays as slices of tensors with a guard of GUARD bytes behind each; the returned function
    counts the guard bytes that have changed."""
    held = {}

    def alloc(nbytes, device=None, stream=None):
        t = torch.full((nbytes + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = (t, nbytes)
        return t.data_ptr()

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", alloc)
    monkeypatch.setattr(torch.cuda, "caching_allocator_delete", lambda p: held.pop(p, None))

    def changed():
        torch.cuda.synchronize()
        return sum(int((t[n:] != 0xA5).sum()) for t, n in held.values())

    return changed


def test_partial_sums_of_many_stored_directions_stay_in_bounds(guarded, monkeypatch):
    """The flexible CG of a mixed solve sums z.Q_j for up to 16 stored directions and 5 time columns from the largest
    number of blocks (more than 1,216 x 256 rows): 80 columns of partials."""
    import paper_1601_07384_gb300 as g
    inner = 5
    monkeypatch.setenv("STDG_MIXED_INNER", str(inner))
    s = g.Solver(g.Mesh(*kuhn_mesh(18, seed=0)), g.Reference(2, 4), 0.01, precision="mixed_f32")
    assert s.ne * s.N > 1216 * 256
    b = torch.randn(s.ne * s.Nst, generator=torch.Generator().manual_seed(1), dtype=torch.float64)
    b[[a * s.N for a in range(s.Ng)]] = 0.0
    x, st = s.solve(b.cuda(), tol=1e-9, method="kron_pcg")
    assert st["iterations"] > 17 * inner             # all 16 slots were used, and the oldest overwritten
    assert st["rel_residual"] <= 1e-9
    assert guarded() == 0
