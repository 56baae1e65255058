"""Fits with the digit split at bonds where its products are large and no multiple of a tile: the partials' sum takes
its 32-row tiles (more than eight to an SM) with remainders in both directions, and 8-row tiles at the chain's ends."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from oracle.mpo import mpo_diff_norm, mpo_norm  # noqa: E402
from paper_2606_23274_gb300 import ttfit  # noqa: E402


@pytest.mark.parametrize("chi", [67, 90])
def test_digit_split_at_ragged_sizes(chi):
    rng = np.random.default_rng(chi)
    bonds = [min(4 ** l, 4 ** (9 - l), chi) for l in range(10)]
    pair = [[rng.standard_normal((bonds[l], 2, 2, bonds[l + 1])) / (2 * bonds[l + 1] ** 0.5) for l in range(9)]
            for _ in range(2)]
    C, n2 = {}, {}
    for precision in ("fp64", "bf16_split"):
        h = ttfit.tt_fit_create(*pair, chi, 0.0, "site", update="rsvd", oversample=6, seed=5, precision=precision,
                                conv_tol=0.0)
        n2[precision] = h.sweep(1)["norm2_C"]
        C[precision] = [c.cpu().numpy() for c in h.result()]
        h.destroy()
    # as for the other double-FP32 fits: contractions to some 1e-14, times what the truncation's gaps magnify
    assert abs(n2["bf16_split"] - n2["fp64"]) <= 1e-10 * n2["fp64"]
    assert mpo_diff_norm(C["bf16_split"], C["fp64"]) <= 1e-9 * mpo_norm(C["fp64"])
