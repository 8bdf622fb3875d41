"""The hop limit of the element search (walk_max) on 2-D FP32 grids: a target that needs more elements keeps
its old value and is counted, on the two-phase kernel (tile configuration 0) as on the tiled one."""
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


@pytest.mark.parametrize("n", [(64, 64), (121, 90)])
def test_walk_limit_is_kept(sl, n):
    rng = np.random.default_rng(3)
    y, x = np.meshgrid(np.arange(n[1]) / n[1], np.arange(n[0]) / n[0], indexing="ij")
    # a shear of slope 1.5 to 4 along x: the refined start misses by several elements
    D = np.stack([6.0 * np.sin(6 * np.pi * y + 1.0), 1.3 + 0.4 * np.sin(2 * np.pi * x)], -1)
    D = torch.tensor(D, dtype=torch.float32, device=DEV)
    f = torch.tensor(rng.standard_normal((3, n[1], n[0])), dtype=torch.float32, device=DEV)
    lost = []
    for walk_max in (1, 2, 3, 4, 5, 64):
        out, diag = [], []
        for cfg in (0, 1):
            g = sl.Grid(2, n, 3, sl.SL_F32, tile_config=cfg, walk_max=walk_max)
            g.set_displacement(D)
            o = torch.empty_like(f)
            g.remap(f, o)
            out.append(o)
            diag.append(g.diagnostics())
        for k in ("targets", "fail_locate", "fail_newton", "fail_fold", "order_hist"):
            assert diag[0][k] == diag[1][k], (walk_max, k, diag)
        assert torch.equal(out[0], out[1])
        lost.append(diag[0]["fail_locate"])
    assert lost[0] > 0 and lost[0] >= lost[1] >= lost[2] and lost[-1] == 0, lost  # the limit takes effect
