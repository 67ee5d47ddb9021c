"""Products r = A x - y, g = A^T r (rows a6-a7, n <= 128) where the kernel's split of
the rows can go wrong: fewer rows than a step of its ring holds, remainders of a step, one
row per block, more rows per block than the prefetched measurements, no measurements.

Tolerance: an entry of r adds N products in chains of at most N/512 <= 32 terms, then
about 10 levels of pairwise sums, so its error is below 42 * 2^-24 * |A||x| = 2.5e-6 |A||x|
(g: chains of at most m/136 + 136/12 terms over the rows, below 600 here); the bounds below
are the ones of the products' other tests, 1e-5 of the absolute sums."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import quant_ref
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tv(cuda_device):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1001_1774_gb300 as tv
    return tv


@pytest.mark.parametrize("prec,n,m,with_y", [
    (0, 16, 7, True), (0, 16, 17, False), (0, 16, 136 * 1024 + 17, True), (0, 32, 5, True),
    (0, 32, 545, False), (0, 48, 3, True), (0, 48, 549, True), (0, 64, 1, True),
    (0, 64, 273, False), (0, 64, 545, True), (0, 96, 137, True), (0, 96, 409, True), (0, 128, 1, True),
    (0, 128, 273, False), (1, 32, 9, True), (1, 64, 547, True), (1, 128, 137, True),
    (2, 32, 545, True), (2, 64, 3, False), (2, 128, 545, True)])
def test_products_at_the_edges_of_the_row_split(tv, prec, n, m, with_y):
    N = n * n
    A = synth.gaussian_matrix(5 + n + prec, m, N)
    Ae = quant_ref.effective_A(A, prec).astype(np.float64)
    rng = np.random.default_rng(1000 * n + m)
    x = rng.standard_normal(N).astype(np.float32)
    y = rng.standard_normal(m).astype(np.float32) if with_y else None
    opt = tv.tvcs_default_options()
    opt.tau = 0.1
    opt.precision = prec
    h = tv.tvcs_create(torch.from_numpy(A).cuda(), 0, m, n, 1.0, 1.0, 0.0, opt)
    r = np.empty(m, np.float32)
    g = np.empty(N, np.float32)
    tv.tvcs_apply(h, x, y, r, g)
    tv.tvcs_destroy(h)
    rr = Ae @ x.astype(np.float64) - (y.astype(np.float64) if with_y else 0.0)
    scale_r = np.abs(Ae) @ np.abs(x.astype(np.float64)) + (np.abs(y) if with_y else 0.0)
    assert np.all(np.abs(r - rr) <= 1e-5 * scale_r + 1e-30)
    gr = Ae.T @ r.astype(np.float64)
    scale_g = np.abs(Ae).T @ np.abs(r.astype(np.float64))
    assert np.all(np.abs(g - gr) <= 1e-5 * scale_g + 1e-30)


@pytest.mark.parametrize("kind,n,m", [("fp32", 16, 77), ("fp32", 96, 921), ("fp8", 64, 701), ("cluster", 192, 500),
                                      ("dct", 48, 461)])
def test_apply_takes_every_kind_of_array(tv, kind, n, m):
    """Arrays that the kernels may use as they are and arrays that go through the handle's buffers
    (host memory, a start that is not 16-byte aligned, a result over an input or next to it)
    give the same bits."""
    N = n * n
    g = torch.Generator(device="cuda").manual_seed(n + m)
    opt = tv.tvcs_default_options()
    opt.tau = 0.1
    if kind == "dct":
        rows = np.random.default_rng(m).choice(N, size=m, replace=False).astype(np.int32)
        h = tv.tvcs_create_partial_dct(rows, n, 1.0, 1.0, 0.0, opt)
    else:
        opt.precision = tv.TVCS_PREC_FP8_BF16 if kind == "fp8" else tv.TVCS_PREC_FP32
        h = tv.tvcs_create(torch.randn(m, N, generator=g, device="cuda") / m ** 0.5, 0, m, n, 1.0, 1.0, 0.0, opt)
    x, y = torch.randn(N, generator=g, device="cuda"), torch.randn(m, generator=g, device="cuda")
    r, gg = torch.empty_like(y), torch.empty_like(x)
    tv.tvcs_apply(h, x, y, r, gg)

    def odd(t):   # the same values from an address that is 4 bytes off
        b = torch.empty(t.numel() + 1, device="cuda")
        b[1:] = t
        return b[1:]

    def check(a, b):
        for p, q in ((a, r), (b, gg)):
            assert np.array_equal(p if isinstance(p, np.ndarray) else p.cpu().numpy(), q.cpu().numpy())

    for xs, ys, ro, go in (
            (x.cpu().numpy(), y, torch.empty_like(y), torch.empty_like(x)),
            (x, y.cpu().numpy(), np.empty(m, np.float32), np.empty(N, np.float32)),
            (odd(x), odd(y), odd(r), odd(gg)), (x, odd(y), odd(r), torch.empty_like(x))):
        tv.tvcs_apply(h, xs, ys, ro, go)
        check(ro, go)
    # results over the inputs
    x2, y2 = x.clone(), y.clone()
    tv.tvcs_apply(h, x2, y2, y2, x2)
    check(y2, x2)
    # r and g in one buffer, g at an aligned place right after r's last entry
    pad = (4 - m % 4) % 4
    b = torch.zeros(pad + m + N, device="cuda")
    tv.tvcs_apply(h, x, y, b[pad:pad + m], b[pad + m:])
    check(b[pad:pad + m], b[pad + m:])
    # no measurements: r = A x
    tv.tvcs_apply(h, x, None, ro_ := torch.empty_like(y), torch.empty_like(x))
    tv.tvcs_apply(h, x.cpu().numpy(), None, rh := np.empty(m, np.float32), np.empty(N, np.float32))
    assert np.array_equal(ro_.cpu().numpy(), rh)
    tv.tvcs_destroy(h)
