"""The FP64 trajectory launch of the swirl over all its angle ranges -- below pi/128, up to pi/16, beyond (where
the general RK4 takes over, for a whole warp or for single nodes), near the flow's turning time and backwards --
against the oracle's trajectories.

Both sides round at 1.1e-16; a stage's error passes through at most three further stages whose strain over the
step is below 4 here (pi dt): 2e-14 of the largest displacement leaves a factor of ten."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(5, 7), (33, 64), (257, 130)])
@pytest.mark.parametrize("t,dt", [(0.1, 1e-3), (0.1, 0.02), (0.1, 0.07), (0.1, 0.125), (0.1, 0.16), (0.3, 0.4),
                                  (2.45, 0.2), (2.5, 1.0), (1.0, -0.15), (0.0, 0.0)])
def test_swirl_trajectories_at_every_angle(n, t, dt):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from oracle import oracle as orc
    from paper_1410_2817_gb300 import sl
    orc.build()
    want = orc.advect(orc.OracleGrid(dim=2, n=n, velocity="swirl2d", velocity_params=[5.0]), t, dt)
    g = sl.Grid(2, n, 1, sl.SL_F64, velocity="swirl2d", velocity_params=[5.0])
    g.advect(t, dt)
    got = g.get_displacement().cpu().numpy().reshape(want.shape)
    assert np.abs(got - want).max() <= 2e-14 * np.abs(want).max()
