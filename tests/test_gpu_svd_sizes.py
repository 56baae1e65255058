"""tt_svd_truncated at the edges of its kernels' size ranges: the FP64 cluster Jacobi with 1, 8 and 16
CTAs (changes at 24 and 96 columns; odd and even blocks; plain rotations up to 300 rows of columns and
accumulated rotations together, scaled ones above)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_23274_gb300 import ttfit  # noqa: E402

EPS = np.finfo(np.float64).eps


@pytest.mark.parametrize("m,n", [(1, 1), (2, 2), (3, 2), (23, 23), (24, 24), (25, 31), (300, 7), (95, 95), (96, 97),
                                 (129, 127), (1, 600), (900, 24), (200, 120), (281, 33)])
@pytest.mark.parametrize("floor", [1e-1, 1e-13])
def test_svd_at_the_edges_of_the_kernels(m, n, floor):
    rng = np.random.default_rng(m * 2000 + n)
    r = min(m, n)
    s = floor ** (np.arange(r) / max(1, r - 1))
    M = (rng.standard_normal((m, r)) * s) @ rng.standard_normal((r, n))
    U, S, Vt, _ = ttfit.tt_svd_truncated(M, chi_max=r, tau_rel=0.0)
    U, S, Vt = U.cpu().numpy(), S.cpu().numpy(), Vt.cpu().numpy()
    # each of at most 60 sweeps rotates a column r - 1 times, with a rounding of eps each
    tol = 60 * r * EPS
    norm = np.linalg.norm(M)
    assert np.linalg.norm(U * S[None, :] @ Vt - M) <= tol * norm
    assert np.abs(U.T @ U - np.eye(r)).max() <= tol and np.abs(Vt @ Vt.T - np.eye(r)).max() <= tol
    assert np.abs(S - np.linalg.svd(M, compute_uv=False)).max() <= tol * norm


@pytest.mark.parametrize("r,floor", [(32, 1e-4), (33, 1e-14), (64, 1e-18), (95, 1e-9), (96, 1e-14), (128, 1e-4), (129, 1e-14),
                                     (193, 1e-6), (256, 1e-3)])
def test_svd_with_fp32_sweeps_is_as_accurate(r, floor):
    """From 32 columns on the early sweeps run in FP32: clustered, graded and rank-deficient spectra still come out
    to FP64 rounding."""
    rng = np.random.default_rng(r)
    s = floor ** (np.arange(r) / (r - 1))
    s[r // 3:r // 3 + 4] = s[r // 3]        # a cluster
    s[-2:] = 0.0                            # rank deficient
    Q1, _ = np.linalg.qr(rng.standard_normal((r, r)))
    Q2, _ = np.linalg.qr(rng.standard_normal((r, r)))
    M = (Q1 * s) @ Q2.T
    U, S, Vt, _ = ttfit.tt_svd_truncated(M, chi_max=r, tau_rel=0.0)
    U, S, Vt = U.cpu().numpy(), S.cpu().numpy(), Vt.cpu().numpy()
    tol = 60 * r * EPS
    k = int(np.sum(s > 1e-9))               # vectors of values above the rounding level of the product M
    assert np.linalg.norm(U * S[None, :] @ Vt - M) <= tol * np.linalg.norm(M)
    assert np.abs(U[:, :k].T @ U[:, :k] - np.eye(k)).max() <= tol
    assert np.abs(Vt[:k] @ Vt[:k].T - np.eye(k)).max() <= tol
    assert np.abs(S - s[np.argsort(-s)]).max() <= tol


@pytest.mark.parametrize("r", [33, 75, 129, 250])
def test_svd_with_fp32_sweeps_repeats_its_bits(r):
    """The kernels add in a fixed order and their lanes agree on every rotation: the same input, the same bits."""
    M = torch.from_numpy(np.random.default_rng(r).standard_normal((r, r))).cuda()
    first = ttfit.tt_svd_truncated(M, chi_max=r, tau_rel=0.0)
    for _ in range(8):
        again = ttfit.tt_svd_truncated(M, chi_max=r, tau_rel=0.0)
        assert all(torch.equal(a, b) for a, b in zip(first[:3], again[:3]))


# one CTA, 8 and 16 CTAs, the long side on either hand; entries whose squares, or their products, leave the range
@pytest.mark.parametrize("m,n", [(24, 16), (64, 40), (40, 64), (130, 120)])
@pytest.mark.parametrize("scale", [1e80, 1e-80, 1e140, 1e-140])
def test_svd_does_not_depend_on_the_scale(m, n, scale):
    rng = np.random.default_rng(m * 2000 + n)
    r = min(m, n)
    M = rng.standard_normal((m, n))
    U, S, Vt, _ = ttfit.tt_svd_truncated(M * scale, chi_max=r, tau_rel=0.0)
    U, S, Vt = U.cpu().numpy(), S.cpu().numpy() / scale, Vt.cpu().numpy()
    tol = 60 * r * EPS  # as above
    assert np.linalg.norm(U * S[None, :] @ Vt - M) <= tol * np.linalg.norm(M)
    assert np.abs(U.T @ U - np.eye(r)).max() <= tol and np.abs(Vt @ Vt.T - np.eye(r)).max() <= tol
    assert np.abs(S - np.linalg.svd(M, compute_uv=False)).max() <= tol * np.linalg.norm(M)


# the same at scales whose squares leave FP64's range altogether, and through the kernel for what fits no cluster; the
# rule has to keep the same rank
@pytest.mark.parametrize("m,n", [(24, 16), (64, 40), (40, 64), (345, 340)])
@pytest.mark.parametrize("scale", [1e200, 1e-200, 1e300, 1e-280])
def test_svd_at_the_ends_of_the_range(m, n, scale):
    rng = np.random.default_rng(m * 2000 + n)
    r = min(m, n)
    M = rng.standard_normal((m, r)) * 10.0 ** -np.linspace(0, 6, r) @ rng.standard_normal((r, n))
    k0 = ttfit.tt_svd_truncated(M, chi_max=r, tau_rel=1e-3)[3]
    U, S, Vt, k = ttfit.tt_svd_truncated(M * scale, chi_max=r, tau_rel=1e-3)
    U, S, Vt = U.cpu().numpy(), S.cpu().numpy() / scale, Vt.cpu().numpy()
    tol = 60 * r * EPS  # as above
    assert k == k0
    assert np.linalg.norm(U * S[None, :] @ Vt - M) <= tol * np.linalg.norm(M)
    assert np.abs(U.T @ U - np.eye(r)).max() <= tol and np.abs(Vt @ Vt.T - np.eye(r)).max() <= tol


@pytest.mark.parametrize("m,n", [(24, 16), (64, 40), (40, 64)])
def test_svd_with_one_very_large_entry(m, n):
    M = np.random.default_rng(0).standard_normal((m, n))
    M[3, 5] = 1e200
    U, S, Vt, k = ttfit.tt_svd_truncated(M, chi_max=min(m, n), tau_rel=0.0)
    assert k == 1 and abs(float(S[0]) / 1e200 - 1) <= 60 * min(m, n) * EPS
    assert bool(torch.isfinite(U).all() and torch.isfinite(S).all() and torch.isfinite(Vt).all())
    assert abs(abs(float(U[3, 0])) - 1) <= 60 * min(m, n) * EPS and abs(abs(float(Vt[0, 5])) - 1) <= 60 * min(m, n) * EPS
    M[:] = 1.7e308  # the largest singular value is not a number of FP64
    with pytest.raises(ttfit.TTError) as e:
        ttfit.tt_svd_truncated(M, chi_max=1, tau_rel=0.0)
    assert e.value.code == ttfit.TT_ERR_NUMERICAL


@pytest.mark.parametrize("m,n", [(24, 16), (40, 64), (120, 100)])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_svd_refuses_what_is_not_finite(m, n, value):
    M = np.random.default_rng(0).standard_normal((m, n))
    M[m // 2, n // 2] = value
    with pytest.raises(ttfit.TTError) as e:
        ttfit.tt_svd_truncated(M, chi_max=min(m, n), tau_rel=0.0)
    assert e.value.code == ttfit.TT_ERR_NUMERICAL


# null columns, null rows, equal columns, the null matrix; one CTA and clusters, the long side on either hand
@pytest.mark.parametrize("m,n", [(24, 16), (33, 32), (64, 40), (40, 64), (130, 120)])
@pytest.mark.parametrize("kind", ["columns", "rows", "rank1", "zero"])
def test_svd_of_a_rank_deficient_matrix(m, n, kind):
    r = min(m, n)
    M = np.random.default_rng(m).standard_normal((m, n))
    if kind == "columns":
        M[:, n // 2:] = 0.0
    elif kind == "rows":
        M[m // 2:] = 0.0
    elif kind == "rank1":
        M[:] = 1.0
    else:
        M[:] = 0.0
    U, S, Vt, k = ttfit.tt_svd_truncated(M, chi_max=r, tau_rel=0.0)
    U, S, Vt = U.cpu().numpy(), S.cpu().numpy(), Vt.cpu().numpy()
    tol = 60 * r * EPS  # as above
    rank = np.linalg.matrix_rank(M)
    assert k == max(rank, 1)
    assert np.linalg.norm(U * S[None, :] @ Vt - M) <= tol * np.linalg.norm(M)
    assert np.abs(S - np.linalg.svd(M, compute_uv=False)).max() <= tol * np.linalg.norm(M)
    square = Vt if m >= n else U.T  # the r x r factor is orthogonal whatever the rank
    assert np.abs(square @ square.T - np.eye(r)).max() <= tol
    long = U[:, :rank] if m >= n else Vt[:rank].T
    assert np.abs(long.T @ long - np.eye(rank)).max(initial=0.0) <= tol
