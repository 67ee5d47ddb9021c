"""tvcs_apply_noalloc with its results over its inputs (r over y, g over x): each block reads the
measurements of its rows before it stores r there, also where they do not fit in its shared
memory (more than 1024 rows a block: m > 139,264), and g is stored when every block has
read x.  Both calls add in the same order, so the bound is equality."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def tv(cuda_device):
    import __graft_entry__
    __graft_entry__.build()
    import paper_1001_1774_gb300 as tv
    return tv


@pytest.mark.parametrize("n,m", [(16, 136 * 1024 + 17), (16, 136 * 1024 + 136 * 16 + 5), (32, 136 * 1025), (16, 77),
                                 (48, 691), (96, 921), (128, 1000)])
def test_results_over_the_inputs(tv, n, m):
    gen = torch.Generator(device="cuda").manual_seed(n + m)
    A = torch.randn(m, n * n, generator=gen, device="cuda") / m ** 0.5
    x, y = torch.randn(n * n, generator=gen, device="cuda"), torch.randn(m, generator=gen, device="cuda")
    r, g = torch.empty_like(y), torch.empty_like(x)
    tv.tvcs_apply_noalloc(A, m, n, x, y, r, g)
    for _ in range(5):
        for over_x in (False, True):
            x2, y2 = x.clone(), y.clone()
            g2 = x2 if over_x else torch.empty_like(x)
            tv.tvcs_apply_noalloc(A, m, n, x2, y2, y2, g2)
            assert torch.equal(y2, r) and torch.equal(g2, g)
