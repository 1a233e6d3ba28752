"""Device memory of a solver comes from its allocator alone, and stdg_get_blocks does without where that has none."""
import ctypes as C

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from inputs import kuhn_mesh
from oracle.blocks import SpaceTimeDG
from oracle.mesh import Mesh


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1601_07384_gb300.build import build
    build()


class PoolHigh:
    """High-water mark of the device's default memory pool (stream-ordered allocations), reset to 0 on entry."""
    USED_MEM_HIGH = 8

    def __init__(self):
        self.cu = C.CDLL("libcuda.so.1")
        self.pool = C.c_void_p()
        assert self.cu.cuDeviceGetDefaultMemPool(C.byref(self.pool), torch.cuda.current_device()) == 0
        zero = C.c_uint64(0)
        assert self.cu.cuMemPoolSetAttribute(self.pool, self.USED_MEM_HIGH, C.byref(zero)) == 0

    def read(self):
        v = C.c_uint64(0)
        assert self.cu.cuMemPoolGetAttribute(self.pool, self.USED_MEM_HIGH, C.byref(v)) == 0
        return v.value


@pytest.mark.parametrize("n,p,pt", [(1, 4, 0), (2, 1, 1), (2, 4, 4), (3, 2, 0)])
def test_get_blocks_takes_memory_from_the_allocator_or_none_and_matches_oracle(n, p, pt, monkeypatch):
    """Nothing from the runtime's pool, and the allocator gets back what it gave; once it gives no more, the same
    values.  (1, 4, 0): the room that the blocks are then decoded in holds a block and a half, so that most pieces
    end inside one."""
    import paper_1601_07384_gb300 as g
    s = g.Solver(g.Mesh(*kuhn_mesh(n, seed=0)), g.Reference(p, pt), 1.0)
    torch.cuda.synchronize()
    high, live = PoolHigh(), s.alloc_stats()[0]
    blk = s.blocks()
    assert high.read() == 0 and s.alloc_stats()[0] == live

    def none_left(*args, **kwargs):
        raise torch.cuda.OutOfMemoryError("none left")

    monkeypatch.setattr(torch.cuda, "caching_allocator_alloc", none_left)
    torch.cuda.synchronize()
    free, calls = torch.cuda.mem_get_info()[0], s.alloc_stats()[1]
    again = s.blocks()
    assert high.read() == 0 and torch.cuda.mem_get_info()[0] == free and s.alloc_stats()[1] == calls
    assert all(np.array_equal(blk[k], again[k]) for k in blk)
    d = SpaceTimeDG(Mesh(*kuhn_mesh(n, seed=0)), p, 0, 1.0)
    B = np.zeros_like(blk["Bdiag"])
    close = lambda a, b: np.abs(a - b).max() <= 1e-12 * max(np.abs(b).max(), 1e-300)   # noqa: E731
    for j in range(d.mesh.nf):
        fb = d.face_blocks(j)
        for k, i in enumerate(fb["sides"]):
            assert close(blk["Q"][j, k], fb["Q"][k]) and close(blk["Mij"][j, k], fb["Mij"][k])
        if d.mesh.interior[j]:
            l, r = fb["sides"]
            assert close(blk["Aoff"][j], -sum(a.T @ b for a, b in zip(*fb["Q"])))
            for k, i in enumerate((l, r)):
                B[i] -= sum(q.T @ q for q in fb["Q"][k])
    assert close(blk["Bdiag"], B)
