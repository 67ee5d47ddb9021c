"""The iteration loop as one persistent launch (n <= 96, stored A) at the sizes where its split
can go wrong: fewer rows of A than blocks of the u-step, one row more or less than the
ring's pieces, rows that do not fit in the ring, one iteration, a run in two parts, a stop by
eq. (stop) -- against the FP64 oracle, and against the same kernels' steps launched one by
one (opt.host_loop).

Tolerance: one iteration in binary32 changes u by at most a few 2^-24 |u| of rounding, and
the iteration is non-expansive (Thm 4), so k <= 40 iterations stay below 40 * 4 * 2^-24 =
1e-5 relative; the stop iteration is the oracle's within one."""
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


def create(tv, P, tau, prec=0, algo=0, max_iter=10, tol=0.0, host_loop=0):
    opt = tv.tvcs_default_options()
    opt.tau, opt.precision, opt.algo, opt.max_iter, opt.host_loop = tau, prec, algo, max_iter, host_loop
    return tv.tvcs_create(torch.from_numpy(P.A).cuda(), 0, P.m, P.n, P.mu, P.beta, tol, opt)


@pytest.mark.parametrize("n,m,prec,algo,iters", [
    (16, 40, 0, 0, 1), (16, 65, 0, 1, 40), (32, 120, 0, 0, 17), (32, 513, 0, 0, 30), (48, 400, 0, 1, 16),
    (48, 609, 0, 0, 40), (64, 700, 0, 0, 31), (64, 1825, 0, 0, 12), (64, 2300, 0, 1, 9), (96, 759, 0, 0, 8),
    (96, 1065, 0, 0, 15), (32, 310, 1, 0, 20), (64, 1217, 1, 0, 10), (32, 310, 2, 1, 20), (64, 2500, 2, 0, 10)])
def test_loop_against_the_oracle_and_the_single_launches(tv, n, m, prec, algo, iters):
    P = synth.make_problem(n, 0.0, 3, 4, 1e3, 10.0, m=m, noise_c=1e-3)
    A = np.ascontiguousarray(quant_ref.effective_A(P.A, prec))
    tau = oracle.default_tau(A)
    ref = oracle.solve(A, P.f, n, P.mu, P.beta, tau, tol=0.0, max_iter=iters, algo=algo)
    out = []
    for host_loop in (0, 1):
        h = create(tv, P, tau, prec, algo, iters, host_loop=host_loop)
        u = np.empty(n * n, np.float32)
        res = tv.tvcs_solve(h, P.f, u)
        assert res.iters == iters and res.status >= 0
        assert rel(u, ref.u) <= 1e-5
        assert abs(res.objective - res.tv - 0.5 * P.mu * res.resid2) <= 1e-9 * abs(res.objective)
        out.append([tv.get_state(h, k) for k in (tv.TVCS_STATE_U, tv.TVCS_STATE_W, tv.TVCS_STATE_LAMBDA)])
        tv.tvcs_destroy(h)
    for a, b in zip(*out):
        assert rel(a, b) <= 1e-5 or np.linalg.norm(b) == 0.0


@pytest.mark.parametrize("n,m", [(32, 307), (96, 921)])
def test_a_run_in_parts_and_handles_side_by_side(tv, n, m):
    P = synth.make_problem(n, 0.0, 5, 4, 1e3, 10.0, m=m, noise_c=1e-3)
    tau = oracle.default_tau(P.A)
    h, k = create(tv, P, tau, max_iter=13), create(tv, P, tau, max_iter=5)
    u, v = np.empty(n * n, np.float32), np.empty(n * n, np.float32)
    tv.tvcs_solve(k, P.f, v)
    tv.tvcs_solve(h, P.f, u)
    tv.tvcs_iterate(k, 1)
    tv.tvcs_iterate(k, 7)
    assert rel(tv.get_state(k, tv.TVCS_STATE_U), u) <= 1e-5
    assert rel(tv.get_state(k, tv.TVCS_STATE_LAMBDA), tv.get_state(h, tv.TVCS_STATE_LAMBDA)) <= 1e-5
    w = np.empty(n * n, np.float32)
    tv.tvcs_solve(h, P.f, w)   # again: the same bits
    assert np.array_equal(u, w)


# (the first input reaches the cap in the oracle as well, the others stop before it)
@pytest.mark.parametrize("n,mu,beta,tol", [(48, 200.0, 10.0, 1e-3), (48, 20.0, 20.0, 1e-2),
                                           (32, 50.0, 20.0, 1e-3), (96, 50.0, 10.0, 1e-2)])
def test_loop_stops_by_the_relative_change(tv, n, mu, beta, tol):
    P = synth.make_problem(n, 0.3, 7, 4, mu, beta)
    tau = oracle.default_tau(P.A)
    ref = oracle.solve(P.A, P.f, n, P.mu, P.beta, tau, tol=tol, max_iter=400)
    h = create(tv, P, tau, max_iter=400, tol=tol)
    u = np.empty(n * n, np.float32)
    res = tv.tvcs_solve(h, P.f, u)
    assert res.stopped_by_tol == ref.info["stopped_by_tol"] and abs(res.iters - ref.info["iters"]) <= 1
    assert rel(u, ref.u) <= (tol if res.stopped_by_tol else 1e-4)   # one iteration more or less moves u by tol


# The partial-DCT encoder's loop (one cluster): every side, one / few / all coefficients in a
# shuffled order, both algorithms, one iteration, a run in parts, a stop by eq. (stop).
@pytest.mark.parametrize("n,m,algo,iters,tol", [
    (16, 76, 0, 20, 0.0), (16, 256, 1, 1, 0.0), (32, 1, 0, 10, 0.0), (32, 511, 1, 30, 0.0), (48, 461, 0, 25, 0.0),
    (64, 2049, 0, 40, 0.0), (96, 921, 1, 17, 0.0), (96, 9216, 0, 8, 0.0), (128, 4915, 0, 40, 0.0),
    (128, 4915, 0, 400, 3e-3), (128, 16383, 0, 5, 0.0)])
def test_dct_loop_against_the_oracle_and_the_single_launches(tv, n, m, algo, iters, tol):
    rng = np.random.default_rng(n + m)
    rows = rng.choice(n * n, size=m, replace=False).astype(np.int32)
    f = synth.measure_dct(rows, synth.phantom(n, 8, 5), 1e-3, 77)
    ref = oracle.solve_dct(rows, f, n, 500.0, 64.0, 1.9, tol=tol, max_iter=iters, algo=algo)
    out = []
    for host_loop in (0, 1):
        opt = tv.tvcs_default_options()
        opt.tau, opt.max_iter, opt.algo, opt.host_loop = 1.9, iters, algo, host_loop
        h = tv.tvcs_create_partial_dct(rows, n, 500.0, 64.0, tol, opt)
        u = np.empty(n * n, np.float32)
        res = tv.tvcs_solve(h, f, u)
        assert res.stopped_by_tol == ref.info["stopped_by_tol"] and abs(res.iters - ref.info["iters"]) <= 1
        assert rel(u, ref.u) <= (1e-5 if tol == 0.0 else tol)
        r = tv.get_state(h, tv.TVCS_STATE_R).astype(np.float64)
        assert abs(res.resid2 - (r * r).sum()) <= 1e-9 * res.resid2
        tv.tvcs_iterate(h, 3)
        tv.tvcs_iterate(h, 1)
        out.append([tv.get_state(h, k) for k in (tv.TVCS_STATE_U, tv.TVCS_STATE_W, tv.TVCS_STATE_LAMBDA)])
        tv.tvcs_destroy(h)
    if tol == 0.0:
        for a, b in zip(*out):
            assert rel(a, b) <= 3e-5 or np.linalg.norm(b) == 0.0


# A on chip (n <= 64): fewer rows than blocks, a row more or less than the registers hold, rows in
# shared memory, and (64, 3500), whose rows do not fit; tau from the power iteration.  The power
# iteration's ||A v||^2 carries about 4 roundings of 2^-24 of every dot product, taken as
# independent over N: well below 1e-5; the two runs then agree as above.
@pytest.mark.parametrize("n,m,prec", [
    (16, 1, 0), (16, 31, 0), (16, 256, 0), (32, 15, 0), (32, 128, 1), (32, 129, 0), (32, 1024, 2), (48, 24, 0),
    (48, 1217, 0), (48, 2304, 0), (64, 31, 0), (64, 257, 2), (64, 1216, 0), (64, 1230, 1), (64, 2600, 0), (64, 3500, 0)])
def test_rows_on_chip_and_the_power_iteration(tv, n, m, prec):
    P = synth.make_problem(n, 0.0, 3, 4, 1e3, 10.0, m=m, noise_c=1e-3)
    A = np.ascontiguousarray(quant_ref.effective_A(P.A, prec))
    tau = oracle.default_tau(A)
    h = create(tv, P, 0.0, prec, 0, 8)
    assert abs(tv.tvcs_get_tau(h) / tau - 1) <= 1e-5
    k = create(tv, P, tv.tvcs_get_tau(h), prec, 0, 8, host_loop=1)
    u, v = np.empty(n * n, np.float32), np.empty(n * n, np.float32)
    a, b = tv.tvcs_solve(h, P.f, u), tv.tvcs_solve(k, P.f, v)
    assert a.iters == b.iters == 8 and rel(u, v) <= 1e-5
    r = tv.get_state(h, tv.TVCS_STATE_R).astype(np.float64)
    assert abs(a.resid2 - (r * r).sum()) <= 1e-9 * a.resid2
