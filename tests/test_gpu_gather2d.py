"""The two-phase 2-D FP32 kernel (tile configuration 0) against the tiled kernel (configuration 1): the
same arithmetic target by target, so the bits agree -- at the edges of its strips and tiles, across the
periodic seam, with displacements of a period and more, and for failing targets."""
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


def _fields(n, nf, seed):
    rng = np.random.default_rng(seed)
    y, x = np.meshgrid(np.arange(n[1]) / n[1], np.arange(n[0]) / n[0], indexing="ij")
    planes = []
    for f in range(nf):
        a, b = rng.uniform(0.2, 0.8, size=2)
        smooth = np.sin(2 * np.pi * (x - a)) * np.cos(2 * np.pi * (y - b))
        planes.append(smooth if f % 2 == 0 else smooth + (np.hypot(x - a, y - b) < 0.25))
    return torch.tensor(np.stack(planes), dtype=torch.float32, device=DEV)


def _displacement(n, kind, seed):
    from paper_1410_2817_gb300 import inputs
    shift = {"seam": (3.3, -2.7), "period": (1.4 * n[0], -1.2 * n[1]), "fold": (0.0, 0.0)}[kind]
    D = inputs.smooth_displacement(n, 0.4, seed, shift=shift)
    if kind == "fold":  # one node far off: the elements around it fold or fail
        D[n[1] // 2, n[0] // 2] += 3.0
    return torch.tensor(D, dtype=torch.float32, device=DEV)


@pytest.mark.parametrize("kind", ["seam", "period", "fold"])
@pytest.mark.parametrize("nf", [1, 2, 3, 4])
@pytest.mark.parametrize("n", [(4, 4), (5, 7), (29, 33), (31, 8), (64, 30), (65, 9), (121, 250)])
def test_two_phase_equals_tiled(sl, n, nf, kind):
    f = _fields(n, nf, 1)
    D = _displacement(n, kind, 2)
    for kw in ({}, {"max_order": 0}, {"limiter_threshold": -1.0}):
        out, diag = [], []
        for cfg in (0, 1):
            g = sl.Grid(2, n, nf, sl.SL_F32, tile_config=cfg, **kw)
            g.set_displacement(D)
            for _ in range(2):  # the second launch finds the first one's counters cleared
                o = torch.full_like(f, 7.0)
                g.remap(f, o)
            out.append(o)
            diag.append(g.diagnostics())
        assert torch.equal(out[0], out[1]), float((out[0] - out[1]).abs().max())
        for k in ("targets", "fail_locate", "fail_newton", "fail_fold", "order_hist"):
            assert diag[0][k] == diag[1][k], (k, diag)
        assert diag[0]["timeouts"] == 0


def test_two_phase_large_and_nan(sl):
    """Several tiles and flag items per CTA (a grid above one wave); a NaN displacement stays with its
    own targets."""
    n = (1100, 803)
    f = _fields(n, 3, 3)
    D = _displacement(n, "seam", 4)
    D[400, 500] = float("nan")
    out = []
    for cfg in (0, 1):
        g = sl.Grid(2, n, 3, sl.SL_F32, tile_config=cfg)
        g.set_displacement(D)
        o = torch.empty_like(f)
        g.remap(f, o)
        out.append(o)
    assert torch.equal(out[0], out[1])


def test_two_phase_streams(sl):
    """Launches on several streams at once share the SMs: none waits on another."""
    n = (1100, 900)
    f = _fields(n, 3, 5)
    grids = [sl.Grid(2, n, 3, sl.SL_F32, velocity="swirl2d", velocity_params=[5.0]) for _ in range(4)]
    outs = [torch.empty_like(f) for _ in grids]
    scr = [torch.empty_like(f) for _ in grids]
    streams = [torch.cuda.Stream() for _ in grids]
    torch.cuda.synchronize()
    for g, o, c, st in zip(grids, outs, scr, streams):
        g.step_out(f, o, 0.1, 0.004, 20, scratch=c, stream=st)
    torch.cuda.synchronize()
    for g, o in zip(grids, outs):
        assert torch.equal(o, outs[0]) and g.diagnostics()["timeouts"] == 0
