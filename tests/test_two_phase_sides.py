"""The two-phase 2-D FP32 step serves grids with both sides of at least 16; below, the tiled kernel does (and
the workspace holds no records).  At the line both give the same bits."""
import numpy as np
import pytest
import torch


def _records(sl, n, nf):
    size = [sl.sl_grid_workspace_bytes(sl.make_desc(2, n, nf, sl.SL_F32, velocity="swirl2d", velocity_params=[5.0],
                                                    tile_config=cfg)) for cfg in (0, 1)]
    assert min(size) > 0
    return size[0] - size[1]


@pytest.mark.parametrize("nf", [1, 3, 4])
def test_narrow_grids_hold_no_records(nf):
    from paper_1410_2817_gb300 import build, sl
    build.build()
    for n in ((4, 4), (15, 16), (16, 15), (4, 1 << 20), (12, 2000), (2000, 12)):
        assert _records(sl, n, nf) == 0, n
    for n in ((16, 16), (16, 100), (100, 16), (2048, 2048)):
        assert _records(sl, n, nf) >= (8 if nf == 1 else 16) * n[0] * n[1], n


@pytest.mark.gpu
@pytest.mark.parametrize("nf", [1, 3, 4])
@pytest.mark.parametrize("n", [(15, 16), (16, 15), (16, 16), (16, 129), (200, 17)])
def test_sides_at_the_line_equal_tiled(n, nf):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1410_2817_gb300 import inputs, sl
    f = torch.tensor(np.random.default_rng(2).standard_normal((nf, n[1], n[0])), dtype=torch.float32, device="cuda")
    for shift in ((1.3, -2.7), (9.3, -7.7), (1.5 * n[0], -0.9 * n[1])):
        D = torch.tensor(inputs.smooth_displacement(n, 0.3, 4, shift=shift), dtype=torch.float32, device="cuda")
        out = []
        for cfg in (0, 1):
            g = sl.Grid(2, n, nf, sl.SL_F32, tile_config=cfg, velocity="swirl2d", velocity_params=[5.0])
            g.set_displacement(D)
            o, s = torch.full_like(f, 7.0), torch.full_like(f, 7.0)
            g.remap(f, o)
            g.step_out(f, s, 0.1, 0.02, 2, scratch=torch.empty_like(f))
            out.append((o, s))
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
