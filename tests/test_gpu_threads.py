"""Several threads that use one solver: every product gives what it gives alone, bit for bit."""
import ctypes as C
import sys
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from inputs import kuhn_mesh

ROUNDS = 4000


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_1601_07384_gb300.build import build
    build()


@pytest.mark.parametrize("p,pt", [(1, 0), (2, 1)])
def test_products_of_four_threads_do_not_mix(p, pt):
    """The products share the array that their input vectors are prepared in; ctypes releases the interpreter's
    lock during a call, so that the calls of the threads overlap on the host."""
    import paper_1601_07384_gb300 as g
    from paper_1601_07384_gb300 import _lib
    s = g.Solver(g.Mesh(*kuhn_mesh(2, seed=0)), g.Reference(p, pt), 0.01)
    s.set_boundary(g.zero())
    lib, h = _lib.load(), s._h
    gen = torch.Generator().manual_seed(1)
    np_, nv = s.ne * s.Nst, s.nf * 3 * s.Nst
    x, x2, F = (torch.randn(n, generator=gen, dtype=torch.float64).cuda() for n in (np_, np_, nv))
    ptr = lambda t: C.c_void_p(t.data_ptr())                                         # noqa: E731
    px, px2, pF = ptr(x), ptr(x2), ptr(F)
    calls = [(lambda o: lib.stdg_pressure_apply(h, px, o, 1), np_),
             (lambda o: lib.stdg_pressure_rhs(h, pF, o, 1), np_),
             (lambda o: lib.stdg_pressure_apply(h, px2, o, 0), np_),
             (lambda o: lib.stdg_velocity_update(h, pF, px2, o), nv)]
    want, outs, ptrs = [], [], []
    for call, n in calls:
        want.append(torch.empty(n, dtype=torch.float64, device="cuda"))
        _lib.check(call(ptr(want[-1])))
        outs.append(torch.empty(ROUNDS, n, dtype=torch.float64, device="cuda"))
        ptrs.append([ptr(o) for o in outs[-1]])
    torch.cuda.synchronize()
    start, status = threading.Barrier(len(calls)), [0] * len(calls)

    def work(k):
        torch.cuda.set_device(0)
        call = calls[k][0]
        start.wait()
        for o in ptrs[k]:
            status[k] |= call(o)

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(calls))]
    interval = sys.getswitchinterval()
    sys.setswitchinterval(1e-6)
    try:
        for t in threads:
            t.start()
        for t in threads:
            t.join()
    finally:
        sys.setswitchinterval(interval)
    torch.cuda.synchronize()
    assert status == [0] * len(calls)
    wrong = [int((outs[k] != want[k]).any(1).sum()) for k in range(len(calls))]
    assert wrong == [0] * len(calls)
