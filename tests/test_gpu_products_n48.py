"""Products at 48 x 48 in binary32, whose steps are 8 rows in two row lanes: fewer rows than a
lane, one row more or less than a step, blocks with unequal steps, several rounds of the ring.

Tolerance: an entry of r adds 12 products in order and then about 10 levels of pairwise sums, an
entry of g at most m/136/2 + 1 + 136/12 terms in order (86 here), both below 2^-24 * 100 of the
absolute sums; the bound is the other products' tests', 1e-5."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tv(cuda_device):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1001_1774_gb300 as tv
    return tv


@pytest.mark.parametrize("m", [1, 4, 5, 9, 136 * 8 - 1, 136 * 8 + 1, 136 * 9, 136 * 24 + 77, 20000])
def test_products_48(tv, m):
    n, N = 48, 48 * 48
    gen = torch.Generator(device="cuda").manual_seed(m)
    A = torch.randn(m, N, generator=gen, device="cuda") / m ** 0.5
    x, y = torch.randn(N, generator=gen, device="cuda"), torch.randn(m, generator=gen, device="cuda")
    opt = tv.tvcs_default_options()
    opt.tau = 0.1
    h = tv.tvcs_create(A, 0, m, n, 1.0, 1.0, 0.0, opt)
    out = []
    for call in range(2):
        r, g = torch.empty_like(y), torch.empty_like(x)
        if call == 0:
            tv.tvcs_apply(h, x, y, r, g)
        else:
            tv.tvcs_apply_noalloc(A, m, n, x, y, r, g)
        Ad = A.double()
        er = (r.double() - (Ad @ x.double() - y.double())).abs()
        eg = (g.double() - Ad.T @ r.double()).abs()
        assert bool((er <= 1e-5 * (Ad.abs() @ x.double().abs() + y.double().abs())).all())
        assert bool((eg <= 1e-5 * (Ad.abs().T @ r.double().abs()) + 1e-30).all())
        out.append((r, g))
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    tv.tvcs_destroy(h)
