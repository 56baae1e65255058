"""tt_mpo_grad at bonds around the edges of the GEMM tiles (16, 32, 64; remainders and single rows), against
a plain PyTorch FP64 evaluation of the same objective."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_23274_gb300 import ttfit  # noqa: E402


def _mpo(bonds, seed, dtype):
    g = torch.Generator().manual_seed(seed)
    return [(torch.randn(bonds[l], 2, 2, bonds[l + 1], generator=g, dtype=torch.float64)
             / (2 * bonds[l + 1] ** 0.5)).to(dtype).cuda() for l in range(len(bonds) - 1)]


def _inner(A, B, X):
    E = torch.ones(1, 1, 1, dtype=torch.float64, device="cuda")
    for a, b, x in zip(A, B, X):
        T = torch.einsum("abc,asux,buty->csxty", E, a, b)
        E = torch.einsum("csxty,cstz->xyz", T, x)
    return E.reshape(())


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("bonds", [(1, 15, 16, 17, 1), (1, 2, 33, 31, 1), (1, 64, 65, 1), (1, 1, 3, 1), (1, 130, 9, 1)])
def test_inner_gradient_around_the_tile_edges(bonds, precision):
    dtype = torch.float64 if precision == "fp64" else torch.float32
    other = [1] + [b + 1 for b in bonds[1:-1]] + [1]
    A, B, X = _mpo(bonds, 1, dtype), _mpo(other, 2, dtype), _mpo(bonds, 3, dtype)
    v, gA, gB = ttfit.tt_mpo_grad(A, B, X, "inner", precision)
    A64, B64, X64 = ([t.double().requires_grad_(True) for t in M] for M in (A, B, X))
    ref = _inner(A64, B64, X64)
    g = torch.autograd.grad(ref, A64 + B64)
    # a chain of at most 5 sites x 4 products, sums of at most 4 x 131 terms each: sqrt(524) roundings a product
    tol = 20 * 23 * torch.finfo(dtype).eps
    for got, want in zip(gA + gB, g):
        assert torch.linalg.norm(got.double() - want) <= tol * torch.linalg.norm(want)
    assert abs(v - ref.item()) <= tol * (abs(ref.item()) + torch.linalg.norm(g[-1]).item() * torch.linalg.norm(B64[-1]).item())
