"""Remaps of the plain kernels (FP64, and FP32 with the plain kernel asked for) on narrow and ragged grids,
whose targets are numbered consecutively instead of in blocks: every target is written once, with the value
that the oracle gives it, at sides around the blocks' widths and at the line between the two numberings."""
import numpy as np
import pytest
import torch

from paper_1410_2817_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1410_2817_gb300 import sl as m
    return m


@pytest.fixture(scope="module")
def orc():
    from oracle import oracle
    oracle.build()
    return oracle


@pytest.mark.parametrize("n", [(4, 1000), (17, 33), (28, 64), (29, 64), (31, 61), (32, 64), (33, 60), (1000, 5), (300, 700),
                               (4, 4, 300), (5, 9, 30), (14, 16, 16), (15, 16, 16), (16, 16, 17), (17, 5, 40), (64, 70, 60)])
@pytest.mark.parametrize("order", [1, 2])
def test_narrow_grids_against_oracle(sl, orc, n, order):
    dim = len(n)
    D = inputs.smooth_displacement(n, 0.3, 5, shift=(1.3, -2.6, 0.4)[:dim])
    og = orc.OracleGrid(dim=dim, n=n, nfields=2, max_order=order, start=orc.START_BACKWARD)
    h = np.random.default_rng(1).standard_normal((2,) + og.shape).cumsum(axis=-1) * 0.1
    ref = orc.remap(og, D, orc.flags(og, h), h)
    assert ref.nfail == 0
    face = np.any(np.minimum(np.abs(ref.xi), np.abs(1.0 - ref.xi)) < 1e-9, axis=-1)
    g = sl.Grid(dim, n, 2, sl.SL_F64, max_order=order, walk_start=sl.SL_START_BACKWARD)
    g.set_displacement(torch.tensor(D, device=DEV))
    hin = torch.tensor(h, device=DEV)
    out = torch.full_like(hin, float("nan"))
    g.remap(hin, out)
    assert g.diagnostics()["targets"] == g.nnodes
    err = np.abs(out.cpu().numpy() - ref.h)[:, ~face]
    assert np.isfinite(err).all() and err.max() <= 1e-12 * np.abs(ref.h).max()
    # FP32 on the plain kernel: all written, and nearly everywhere within FP32 of the FP64 result (a limiter
    # flag or a face may fall the other way)
    g = sl.Grid(dim, n, 2, sl.SL_F32, max_order=order, kernel=sl.SL_KERNEL_GENERIC)
    g.set_displacement(torch.tensor(D, dtype=torch.float32, device=DEV))
    out = torch.full_like(hin, float("nan"), dtype=torch.float32)
    g.remap(hin.float(), out)
    assert g.diagnostics()["targets"] == g.nnodes
    err = np.abs(out.double().cpu().numpy() - ref.h)
    assert np.isfinite(err).all() and np.mean(err > 1e-4) <= 0.02
