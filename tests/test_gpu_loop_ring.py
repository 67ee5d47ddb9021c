"""The iteration loop whose rows of A come through the shared-memory ring (k_loop): one case for
every row of its shape table.  Up to 64 x 64 the ring is used just where the rows no
longer fit on chip, which on 152 SMs is above 247, 61, 31, 21 rows a block at n = 16, 32, 48, 64.

Tolerance: as for the loop's other sizes, one iteration in binary32 changes u by at most a few
2^-24 |u| of rounding, and the iteration is non-expansive (Thm 4), so k <= 40 iterations stay
below 40 * 4 * 2^-24 = 1e-5 relative.  (Only u is compared: lambda carries beta.)"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle
import quant_ref
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tv(cuda_device):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1001_1774_gb300 as tv
    return tv


def rel(a, b):
    a, b = np.asarray(a, np.float64).ravel(), np.asarray(b, np.float64).ravel()
    return np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300)


def create(tv, P, tau, prec=0, algo=0, iters=10, host_loop=0, timeout_cycles=0):
    opt = tv.tvcs_default_options()
    opt.tau, opt.precision, opt.algo, opt.max_iter, opt.host_loop = tau, prec, algo, iters, host_loop
    opt.timeout_cycles = timeout_cycles
    return tv.tvcs_create(torch.from_numpy(P.A).cuda(), 0, P.m, P.n, P.mu, P.beta, 0.0, opt)


@pytest.mark.parametrize("n,m,prec,algo,iters", [
    (16, 152 * 247 + 1, 0, 0, 9), (32, 152 * 61 + 1, 0, 0, 10), (32, 152 * 62 + 7, 1, 0, 7), (32, 152 * 63, 2, 1, 8),
    (48, 152 * 31 + 1, 0, 0, 11), (64, 152 * 21 + 1, 0, 1, 8), (64, 152 * 21 + 9, 1, 0, 9), (64, 152 * 22 + 5, 2, 0, 10),
    (96, 761, 0, 0, 7), (16, 152 * 247 + 1, 0, 1, 1)])
def test_ring_against_the_oracle_and_the_single_launches(tv, n, m, prec, algo, iters):
    P = synth.make_problem(n, 0.0, 3, 4, 1e3, 10.0, m=m, noise_c=1e-3)
    A = np.ascontiguousarray(quant_ref.effective_A(P.A, prec))
    tau = oracle.default_tau(A)
    ref = oracle.solve(A, P.f, n, P.mu, P.beta, tau, tol=0.0, max_iter=iters, algo=algo)
    us = []
    for host_loop in (0, 1):
        h = create(tv, P, tau, prec, algo, iters, host_loop)
        u = np.empty(n * n, np.float32)
        res = tv.tvcs_solve(h, P.f, u)
        assert res.iters == iters and res.status >= 0
        assert rel(u, ref.u) <= 1e-5
        r = tv.get_state(h, tv.TVCS_STATE_R).astype(np.float64)
        assert abs(res.resid2 - (r * r).sum()) <= 1e-9 * res.resid2
        us.append(u)
        if host_loop == 0:   # again: the same bits
            v = np.empty(n * n, np.float32)
            tv.tvcs_solve(h, P.f, v)
            assert np.array_equal(u, v)
        tv.tvcs_destroy(h)
    assert rel(us[0], us[1]) <= 1e-5


# A wait that gives up while copies into the ring are in flight, and A on chip: the arrivals that
# the u-step's blocks wait for never come, the call reports it, the next one is right.
@pytest.mark.parametrize("n,m", [(96, 2765), (64, 152 * 21 + 1), (48, 152 * 31 + 1), (64, 1229), (16, 77)])
def test_a_held_loop_times_out_and_the_handle_is_usable(tv, n, m):
    P = synth.make_problem(n, 0.0, 3, 4, 1e3, 10.0, m=m, noise_c=1e-3)
    tau = oracle.default_tau(P.A)
    h, k = create(tv, P, tau, timeout_cycles=10_000_000), create(tv, P, tau)
    u, v = np.empty(n * n, np.float32), np.empty(n * n, np.float32)
    tv.tvcs_test_hold_grid_barrier(h, 1)
    with pytest.raises(tv.TvcsError) as ei:
        tv.tvcs_solve(h, P.f, u)
    assert ei.value.status == tv.TVCS_ERR_TIMEOUT
    tv.tvcs_test_hold_grid_barrier(h, 0)
    assert tv.tvcs_solve(h, P.f, u).iters == tv.tvcs_solve(k, P.f, v).iters == 10
    assert np.array_equal(u, v)
    tv.tvcs_destroy(h)
    tv.tvcs_destroy(k)
