"""Handles used by several host threads at once, each on a stream of its own: the persistent
loops, the chain of launches, the power iteration of tvcs_create and the products share the
device, and every call gives the bits that it gives alone."""
import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tv(cuda_device):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1001_1774_gb300 as tv
    return tv


@pytest.mark.parametrize("sizes", [[(64, 1229), (64, 1229)], [(96, 921), (64, 1229), (48, 691)],
                                   [(16, 77), (32, 307), (96, 2765)], [(128, 1000), (64, 1229), (16, 77)]])
def test_calls_from_several_threads_give_the_bits_of_calls_in_turn(tv, sizes):
    rng = np.random.default_rng(5)
    data = [(torch.randn(m, n * n, device="cuda") / m ** 0.5, rng.standard_normal(m).astype(np.float32))
            for n, m in sizes]
    torch.cuda.synchronize()

    def work(i, rounds, out):
        (n, m), (A, f) = sizes[i], data[i]
        opt = tv.tvcs_default_options()
        opt.max_iter, opt.power_iters = 60, 20
        try:
            for _ in range(rounds):
                h = tv.tvcs_create(A, 0, m, n, 1e3, 10.0, 0.0, opt)
                for _ in range(3):
                    u, r, g = np.empty(n * n, np.float32), np.empty(m, np.float32), np.empty(n * n, np.float32)
                    res = tv.tvcs_solve(h, f, u)
                    tv.tvcs_apply(h, u, f, r, g)
                    out.append((u, r, g, res.iters, res.objective, tv.tvcs_get_tau(h)))
                tv.tvcs_destroy(h)
        except Exception as e:   # the thread's failure is the test's
            out.append(e)

    alone, together = [[] for _ in sizes], [[] for _ in sizes]
    for i in range(len(sizes)):
        work(i, 1, alone[i])
    threads = [threading.Thread(target=work, args=(i, 8, together[i])) for i in range(len(sizes))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for a, b in zip(alone, together):
        for e in a + b:
            if isinstance(e, Exception):
                raise e
        assert len(b) == 24
        for got in b:
            for x, y in zip(got, a[0]):
                assert np.array_equal(x, y)
