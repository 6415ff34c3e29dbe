"""The radix sort at the sizes where its single-launch forms begin and end: a
warp, one block's 1024 and 4096 keys, one cluster's rows and the most it takes,
with 64-bit keys.  Seen through the step network's crowding feature, which
counts the semi-major axes within 50 km in the sorted axes."""
import numpy as np
import pytest
import torch

import population as P

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 31, 33, 1023, 1025, 4096, 4097, 16383, 16385, 163839, 163840,
                               163841, 262145, 400001])
def test_crowding_counts_in_sorted_axes(n):
    from paper_1901_10475_gb300 import stepnet
    torch.cuda.set_device(0)
    els = P.catalog_mixture(n, seed=1200 + n, crossing_frac=0.0)
    # ties in every digit: runs of equal axes, and the order reversed
    els[:, 0] = np.round(els[::-1, 0], 1)
    els[:, 1] = 0.0
    a = els[:, 0]
    s = np.sort(a)
    want = np.log1p(np.searchsorted(s, a + 50.0, "right") - np.searchsorted(s, a - 50.0, "left")
                    - 1.0)
    got = stepnet.features(els)[:, 7].cpu().numpy()
    assert np.abs(got - want).max() <= 1e-6 * (1.0 + np.abs(want).max())
