"""The persistent loop's exchange words carry a 32-bit tag that grows by max_iter with every run.
A handle without a cap (max_iter = 2^31 - 1, a tolerance) comes to the end of the tags with its
third run: no word of an earlier run, and no word that was never written, may then be taken
for one that has arrived.  Equal runs give equal bits, so the bound is equality with a new
handle's first run."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tv(cuda_device):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1001_1774_gb300 as tv
    return tv


@pytest.mark.parametrize("n,m", [(16, 77), (32, 307), (48, 691), (64, 700), (96, 921)])
def test_runs_without_a_cap_agree_past_the_last_tag(tv, n, m):
    P = synth.make_problem(n, 0.0, 7, 4, 20.0, 20.0, m=m, noise_c=1e-3)
    zero = np.zeros(m, np.float32)
    opt = tv.tvcs_default_options()
    opt.tau, opt.max_iter = oracle.default_tau(P.A), 2**31 - 1

    def create():
        return tv.tvcs_create(torch.from_numpy(P.A).cuda(), 0, m, n, P.mu, P.beta, 1e-2, opt)

    def solve(h, f):
        u = np.empty(n * n, np.float32)
        res = tv.tvcs_solve(h, f, u)
        assert res.stopped_by_tol == 1
        return u, res.iters, res.objective

    h = create()
    u, iters, obj = solve(h, P.f)
    assert iters > 4
    for _ in range(3):
        v, it, o = solve(h, P.f)
        assert it == iters and o == obj and np.array_equal(u, v)
    tv.tvcs_destroy(h)
    # runs of one iteration leave the words of every even iteration as they were made
    h = create()
    for _ in range(2):
        v, it, _ = solve(h, zero)
        assert it == 1 and not v.any()
    v, it, o = solve(h, P.f)
    assert it == iters and o == obj and np.array_equal(u, v)
    tv.tvcs_destroy(h)
