"""The fluence solve on grids that end the multigrid hierarchy in every way:
halving down to a few cells, stopping at an odd extent of a few hundred,
a few thousand or more cells, uneven extents, one and several problems; 2D
and 3D, against the oracle's sparse direct solve.

The bound is that of the other fluence tests: the conjugate gradients stop at a
relative residual of 1e-13, which the condition number of these systems
(below 1e4) turns into less than 1e-9 of the solution."""
import numpy as np
import pytest

import phantoms
from oracle import optics
from gpu_helpers import rel_l2, to_gpu, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def solve(shape, pml, batch, seed):
    from paper_1810_11685_gb300.binding import Context
    rng = np.random.default_rng(seed)
    dim, dx = len(shape), 1e-4
    full = tuple(n + 2 * pml for n in shape)
    kappa = 1e-3 / dim * rng.uniform(0.5, 1.5, shape)
    mu = rng.uniform(100.0, 400.0, (batch,) + shape)
    half = min(shape) / 2 * dx * 0.5
    sensors = np.full((2, dim), 0.0)
    sensors[1] = half
    ctx = Context(np.full(full, 1500.0), np.full(full, 1000.0), None, kappa, sensors, dx=dx, dt=0.3 * dx / 1500, nt=4,
                  pml=pml, lossless=True, precision="fp64", max_batch=batch)
    got = to_np(ctx.da_solve(to_gpu(mu, torch.float64), 0b01))
    again = to_np(ctx.da_solve(to_gpu(mu[:1], torch.float64), 0b01))
    assert np.array_equal(again[0], got[0])              # a problem's bits do not depend on the batch
    for b in range(batch):
        assert rel_l2(got[b], optics.fluence(mu[b], kappa, dx, 0b01)) <= 1e-9


@pytest.mark.parametrize("shape,pml", [((64, 64), 8), ((22, 26), 7), ((46, 46), 9), ((50, 94), 7), ((186, 186), 12),
                                       ((12, 80), 10), ((8, 8), 4), ((4, 6), 6)])
@pytest.mark.parametrize("batch", [1, 3])
def test_levels_2d(shape, pml, batch):
    solve(shape, pml, batch, 11 * shape[0] + shape[1])


@pytest.mark.parametrize("shape,pml", [((16, 16, 16), 4), ((18, 18, 18), 3), ((10, 12, 22), 3), ((26, 22, 18), 5)])
def test_levels_3d(shape, pml):
    solve(shape, pml, 2, sum(shape))
