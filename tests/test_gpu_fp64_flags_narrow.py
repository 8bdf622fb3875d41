"""FP64 2-D jump flags on grids of a few columns, around the width below which the plain flag kernel serves:
the criterion itself in numpy, bit for bit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(4, 9), (7, 33), (8, 8), (8, 33), (9, 300)])
def test_flags_of_narrow_grids(n):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1410_2817_gb300 import sl
    h = np.round(np.random.default_rng(n[0]).standard_normal((3, n[1], n[0])) * 8) / 8  # ties at 0.25 among them
    want = np.zeros(h.shape[1:], np.uint8)
    for f in range(3):
        for a in (0, 1):
            dp, dm = np.roll(h[f], -1, a) - h[f], h[f] - np.roll(h[f], 1, a)
            want |= (np.abs(dp - dm) > 0.25 * np.maximum(np.abs(dp), np.abs(dm))).astype(np.uint8) << f
    g = sl.Grid(2, n, 3, sl.SL_F64, limiter_threshold=0.25)
    assert np.array_equal(g.flags(torch.tensor(h, device="cuda")).cpu().numpy(), want)
