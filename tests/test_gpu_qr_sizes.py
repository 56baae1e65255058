"""The Householder QR of the input preparation at the edges of its kernels' size ranges, through
tt_mpo_compress of chains that lose nothing: every site is factorised as a (bond d d') x bond matrix.
FP64 arithmetic (precision fp64) and double-FP32 (precision df32)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from mpo_props import diff_norm, norm2  # noqa: E402
from paper_2606_23274_gb300 import ttfit  # noqa: E402
from paper_2606_23274_gb300.synth import kron_sum_mpo  # noqa: E402


def _dense(cores):
    T = np.ones((1, 1))
    for c in cores:
        T = (T @ c.reshape(c.shape[0], -1)).reshape(-1, c.shape[3])
    return T.reshape(-1)


# legs and bonds; the QR shapes that are the point of each: 1 x 2 .. 2 x 1; 64 x 64, 256 x 128, 512 x 64;
# 512 x 128; 44 x 33, 132 x 90, 360 x 63 (ragged); 81 x 81, 729 x 113; 208 x 64, 1024 x 29
@pytest.mark.parametrize("d,bonds", [((1, 2), (1, 2, 1, 2, 1)), ((2, 2), (1, 4, 16, 64, 128, 64, 16, 4, 1)),
                                     ((2, 2), (1, 4, 16, 64, 128, 128, 64, 16, 4, 1)),
                                     ((2, 2), (1, 3, 11, 33, 90, 63, 16, 4, 1)), ((3, 3), (1, 9, 81, 113, 81, 9, 1)),
                                     ((4, 4), (1, 13, 64, 29, 13, 1))])
@pytest.mark.parametrize("precision,eps", [("fp64", 2.0 ** -52), ("df32", 2.0 ** -44)])
@pytest.mark.parametrize("null", [False, True])
def test_preparation_qr_at_the_edges_of_the_kernels(d, bonds, precision, eps, null):
    rng = np.random.default_rng(sum(bonds))
    L = len(bonds) - 1
    X = [rng.standard_normal((bonds[l], *d, bonds[l + 1])) / bonds[l] ** 0.5 for l in range(L)]
    if null:
        for l in range(1, L - 1):       # a null column and a multiple of another
            if bonds[l + 1] > 2:
                X[l][:, :, :, 1] = 0.0
                X[l][:, :, :, 2] = X[l][:, :, :, 0] * 2.0
    C = ttfit.tt_mpo_compress([torch.from_numpy(x).cuda() for x in X], max(bonds), 0.0, precision=precision)
    got, want = _dense([c.cpu().numpy() for c in C]), _dense(X)
    # each site: at most 60 sweeps of r rotations, or r reflections, of eps each; twice (preparation, compression)
    assert np.linalg.norm(got - want) <= 2 * L * 60 * max(bonds) * eps * np.linalg.norm(want)


# the register kernels' FP64 and double-FP32 forms; an entry that is not finite, or whose square overflows, in the
# column that the first reflector of its site is formed from
@pytest.mark.parametrize("precision", ["fp64", "tf32x3"])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), 1e200])
def test_non_finite_core_is_refused(precision, value):
    rng = np.random.default_rng(3)
    bonds = (1, 4, 16, 32, 32, 16, 4, 1)
    A, B = ([rng.standard_normal((bonds[l], 2, 2, bonds[l + 1])) / bonds[l] ** 0.5 for l in range(7)] for _ in range(2))
    A[3][0, 0, 0, 0] = value
    A, B = ([torch.from_numpy(x).cuda() for x in X] for X in (A, B))
    with pytest.raises(ttfit.TTError) as e:
        f = ttfit.tt_fit_create(A, B, 16, 0.0, "site", precision=precision)
        try:
            f.sweep(1)
        finally:
            f.destroy()
    assert e.value.code == ttfit.TT_ERR_NUMERICAL


def _norm2_of_a_sweep(A, B, chi, precision):
    f = ttfit.tt_fit_create(A, B, chi, 0.0, "site", update="rsvd", oversample=10, seed=0, precision=precision, conv_tol=0.0)
    n2 = f.sweep(1)["norm2_C"]
    f.destroy()
    return n2


# bond weights 2^-k and 0.7^k: what is left of the last columns of a site lies between 4e-23 and 5e-20, where the
# square is in the range of FP32 and its reciprocal is not
@pytest.mark.parametrize("L,K,decay", [(20, 64, 0.5), (30, 128, 0.7)])
def test_graded_chains_are_prepared(L, K, decay):
    A, B = ([torch.from_numpy(x).cuda() for x in kron_sum_mpo(L, K, 0, w, decay=decay)] for w in (0, 1))
    C = ttfit.tt_mpo_compress(A, K, 0.0, precision="df32")
    assert diff_norm(C, A) <= 2 * L * 60 * K * 2.0 ** -44 * norm2(A) ** 0.5  # as above
    want = _norm2_of_a_sweep(A, B, K, "fp64")
    for precision, eps in (("df32", 2.0 ** -44), ("tf32x3", 2.0 ** -21)):
        assert abs(_norm2_of_a_sweep(A, B, K, precision) - want) <= 2 * (2 * L * 60 * K * eps) * want


# a site whose columns all have squares below or above what FP32 holds, or lie themselves outside of it; below, it came
# out as a site without rank
@pytest.mark.parametrize("scale", [2.0 ** -66, 2.0 ** -100, 2.0 ** 66, 2.0 ** 100, 2.0 ** -200, 2.0 ** -450, 2.0 ** 300])
def test_preparation_does_not_depend_on_the_scale_of_a_site(scale):
    A, B = ([torch.from_numpy(x).cuda() for x in kron_sum_mpo(12, 32, 0, w)] for w in (0, 1))
    want = _norm2_of_a_sweep(A, B, 32, "df32")
    A[0] = A[0] * scale
    assert abs(_norm2_of_a_sweep(A, B, 32, "df32") - want * scale ** 2) <= 2 * (2 * 12 * 60 * 32 * 2.0 ** -44) * want * scale ** 2


# columns whose squares are not normal FP64 numbers, or zero
@pytest.mark.parametrize("e", [525, 600, 900])
def test_preparation_takes_sites_whose_squares_underflow(e):
    A, B = ([torch.from_numpy(x).cuda() for x in kron_sum_mpo(12, 32, 0, w)] for w in (0, 1))
    A[0] = A[0] * 2.0 ** -e
    f = ttfit.tt_fit_create(A, B, 32, 0.0, "site", update="rsvd", oversample=10, seed=0, precision="fp64", conv_tol=0.0)
    f.sweep(1)
    C = f.result(torch.float64)
    f.destroy()
    centre = min(range(12), key=lambda l: float(C[l].abs().max()))
    C[centre] = C[centre] * 2.0 ** e
    A[0] = A[0] * 2.0 ** e
    want = _norm2_of_a_sweep(A, B, 32, "fp64")
    assert abs(norm2(C) - want) <= 2 * (2 * 12 * 60 * 32 * 2.0 ** -52) * want
