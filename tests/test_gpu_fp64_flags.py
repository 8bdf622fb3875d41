"""The FP64 2-D jump flags decide in FP32 where that is safe: against the criterion itself in FP64 numpy on
values where it is not -- differences below and above the FP32 range, exact ties at the threshold,
plateaus with rounding noise, infinities and NaN -- at the edges of the kernel's 31-column strips."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1410_2817_gb300 import sl as m
    return m


def _expected(h, thr):
    out = np.zeros(h.shape[1:], np.uint8)
    with np.errstate(all="ignore"):
        for f in range(h.shape[0]):
            hit = np.zeros(h.shape[1:], bool)
            for a in (0, 1):
                dp, dm = np.roll(h[f], -1, a) - h[f], h[f] - np.roll(h[f], 1, a)
                hit |= np.abs(dp - dm) > thr * np.fmax(np.abs(dp), np.abs(dm))
            out |= hit.astype(np.uint8) << f
    return out


@pytest.mark.parametrize("thr", [0.25, 0.0, 3.0])
@pytest.mark.parametrize("n", [(4, 4), (31, 9), (32, 8), (63, 17), (300, 260)])
def test_fp64_flags_special_values(sl, n, thr):
    rng = np.random.default_rng(n[0])
    shape = (n[1], n[0])
    h = np.stack([
        rng.standard_normal(shape).cumsum(axis=1) * 0.1,
        np.round(rng.standard_normal(shape) * 4) / 4,                    # exact ties at 0.25 and plateaus
        1.0 + rng.integers(-1, 2, shape) * 2.0 ** -52,                   # rounding noise
        rng.standard_normal(shape) * 10.0 ** rng.integers(-310, -25, shape),
        rng.standard_normal(shape) * 10.0 ** rng.integers(25, 300, shape),
        np.where(rng.uniform(size=shape) < 0.05, np.inf, rng.standard_normal(shape)),
        np.where(rng.uniform(size=shape) < 0.05, np.nan, rng.standard_normal(shape)),
    ])
    g = sl.Grid(2, n, h.shape[0], sl.SL_F64, limiter_threshold=thr)
    got = g.flags(torch.tensor(h, device="cuda")).cpu().numpy()
    assert np.array_equal(got, _expected(h, thr))
