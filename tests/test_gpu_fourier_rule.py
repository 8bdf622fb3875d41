"""Trajectories of 2-D Fourier velocities in FP32 at both sides of the rules that choose their code (the turn of
the shortest wave in a step; the launch's size): against FP64 trajectories, and a grid alone against the same
grid in a batch, bit for bit."""
import numpy as np
import pytest
import torch

from paper_1410_2817_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sl():
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_1410_2817_gb300 import sl as m
    return m


def _step_of_turn(p, turn):
    """The dt at which the shortest wave turns by `turn` at the root-mean-square speed."""
    m = np.array(p[1:]).reshape(-1, 4)
    k2 = m[:, 0] ** 2 + m[:, 1] ** 2
    speed = 2 * np.pi * np.sqrt((k2 * (m[:, 2] ** 2 + m[:, 3] ** 2)).sum() / 2)
    return turn / (2 * np.sqrt(k2.max()) * speed)


# FP32 phases are good to 2e-6 for |k| <= 4 per axis; the strain over a step of half a turn amplifies that less
# than fivefold: 1e-5 of the largest displacement, doubled.
@pytest.mark.parametrize("turn", [0.05, 0.19, 0.21, 0.5, -0.19])
@pytest.mark.parametrize("modes", [1, 2, 3, 4, 5, 6, 7, 8])
@pytest.mark.parametrize("n", [(9, 7), (130, 61), (513, 511)])
def test_trajectories_at_the_line(sl, n, modes, turn):
    p = inputs.fourier2d_params(np.random.default_rng(modes), modes)
    dt = _step_of_turn(p, turn)
    D = []
    for dtype in (sl.SL_F32, sl.SL_F64):
        g = sl.Grid(2, n, 1, dtype, velocity="fourier2d", velocity_params=p)
        g.advect(0.0, dt)
        D.append(g.get_displacement().double())
    assert float((D[0] - D[1]).abs().max()) <= 2e-5 * float(D[1].abs().max())


@pytest.mark.parametrize("turn", [0.1, 0.19, 0.21])
@pytest.mark.parametrize("modes", [1, 3, 6, 8])
def test_alone_equals_batch(sl, modes, turn):
    p = inputs.fourier2d_params(np.random.default_rng(modes), modes)
    dt = _step_of_turn(p, turn)
    sides = [(33, 40), (100, 64), (530, 520)]

    def fields(n):
        return torch.tensor(np.random.default_rng(n[0]).standard_normal((2, n[1], n[0])), dtype=torch.float32, device="cuda")

    def grid(n):
        return sl.Grid(2, n, 2, sl.SL_F32, velocity="fourier2d", velocity_params=p, tile_config=1)

    together = [fields(n) for n in sides]
    batch = sl.Batch([grid(n) for n in sides], together, [torch.empty_like(f) for f in together], [0.0] * 3, [dt] * 3)
    batch.step(3)
    torch.cuda.synchronize()
    for n, b in zip(sides, together):
        a = fields(n)
        grid(n).step(a, torch.empty_like(a), 0.0, dt, 3)
        assert torch.equal(a, b), n
