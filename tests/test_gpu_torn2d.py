"""2-D FP32 fields torn at the seam by a solid-body rotation: the two-phase kernel's failing and re-solved
targets against the tiled kernel's, bit for bit and count by count, at the walks' full length and cut short.
(Where a tile's window does not fit shared memory the tiled kernel searches from unrefined starts; in a torn
map that may end in another element or in none: there only the failures are compared, which are no more.)"""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walk_max", [0, 3, 10])
@pytest.mark.parametrize("n,angle", [((64, 64), 0.2), ((96, 130), 0.06), ((384, 384), 0.03), ((64, 64), 0.8)])
@pytest.mark.parametrize("nf", [1, 3])
def test_torn_fields_equal_tiled(n, angle, nf, walk_max):
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1410_2817_gb300 import sl
    y, x = torch.meshgrid(torch.arange(n[1]) / n[1], torch.arange(n[0]) / n[0], indexing="ij")
    f = torch.stack([torch.sin(6.0 * x + k * y) + (x > 0.5) * (k % 2) for k in range(nf)]).float().cuda().contiguous()
    out, diag = [], []
    for cfg in (0, 1):
        g = sl.Grid(2, n, nf, sl.SL_F32, velocity="solid_body", velocity_params=[1.0, 0.5, 0.5], tile_config=cfg,
                    walk_max=walk_max)
        o = torch.full_like(f, 7.0)
        g.step_out(f, o, 0.0, angle, 1)
        out.append(o)
        diag.append(g.diagnostics())
    assert diag[0]["targets"] == diag[1]["targets"] and diag[0]["newton_f64"] > 0
    if diag[1]["tiles_fallback"]:
        failed = [d["fail_locate"] + d["fail_newton"] + d["fail_fold"] for d in diag]
        assert failed[0] <= failed[1]
        return
    assert torch.equal(out[0], out[1])
    for k in ("fail_locate", "fail_newton", "fail_fold", "newton_f64", "order_hist", "hops_sum", "iters_sum"):
        assert diag[0][k] == diag[1][k], (k, diag)
