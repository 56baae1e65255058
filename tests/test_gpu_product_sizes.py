"""tt_mpo_naive_product at ragged sizes: rows whose length is and is not a multiple of 16 bytes, single
columns, more sites than one launch takes, unequal legs. Exact up to one rounding a term."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_23274_gb300 import ttfit  # noqa: E402


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("L,a,b,s,u,t", [(1, 1, 1, 3, 2, 5), (3, 1, 2, 2, 2, 2), (4, 5, 7, 2, 3, 1), (3, 33, 31, 2, 2, 2),
                                         (40, 2, 3, 2, 1, 2), (3, 16, 24, 1, 4, 3)])
def test_product_at_ragged_sizes(dtype, L, a, b, s, u, t):
    g = torch.Generator().manual_seed(L * 100 + a)
    bond = lambda c, l: 1 if l in (0, L) else c + (l % 2)
    A = [torch.randn(bond(a, l), s, u, bond(a, l + 1), generator=g, dtype=torch.float64).to(dtype).cuda() for l in range(L)]
    B = [torch.randn(bond(b, l), u, t, bond(b, l + 1), generator=g, dtype=torch.float64).to(dtype).cuda() for l in range(L)]
    for x, y, c in zip(A, B, ttfit.tt_mpo_naive_product(A, B)):
        want = torch.einsum("isuj,kutl->ikstjl", x.double(), y.double()).reshape(c.shape)
        size = torch.einsum("isuj,kutl->ikstjl", x.double().abs(), y.double().abs()).reshape(c.shape)
        assert ((c.double() - want).abs() <= u * torch.finfo(dtype).eps * size).all()
