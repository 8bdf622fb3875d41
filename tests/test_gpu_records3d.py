"""3-D FP32 launches that read their taps from records (fused steps of up to four fields, plain remaps of
three and four) against the launches that gather from the planes (tile configuration 1): the same sums on
the same values, bit for bit, at the smallest sides, odd sides and across the periodic seam."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1410_2817_gb300 import sl as m
    return m


@pytest.mark.parametrize("nf", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [(4, 4, 4), (5, 7, 6), (29, 33, 9), (31, 16, 40)])
def test_records_equal_planes(sl, n, nf):
    from paper_1410_2817_gb300 import inputs
    rng = np.random.default_rng(nf)
    h = rng.standard_normal((nf, n[2], n[1], n[0])).cumsum(axis=3) * 0.1
    h[nf - 1] = np.where(h[nf - 1] > 0, 1.0, h[nf - 1])
    f = torch.tensor(h, dtype=torch.float32, device=DEV)
    D = torch.tensor(inputs.smooth_displacement(n, 0.3, 3, shift=(2.6, -3.2, 1.7)), dtype=torch.float32, device=DEV)
    for kw in ({}, {"max_order": 0}, {"limiter_threshold": -1.0}):
        res = []
        for cfg in (0, 1):
            g = sl.Grid(3, n, nf, sl.SL_F32, velocity="uniform", velocity_params=[0.13, -0.21, 0.08], tile_config=cfg, **kw)
            g.set_displacement(D)
            remapped, stepped = torch.empty_like(f), torch.empty_like(f)
            g.remap(f, remapped)
            g.step_out(f, stepped, 0.0, 0.5, 2, scratch=torch.empty_like(f))  # fused launches
            res.append((remapped, stepped, g.diagnostics()["order_hist"]))
        assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
        assert res[0][2] == res[1][2]
