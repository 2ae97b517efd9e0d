"""The whole-loop kernel of small 2D FP32 grids against the launched generic
passes (generic_fft contexts) on the same inputs: every square extent with a
kernel of its own, uneven grids on the kernel for runtime lengths, row and
column blocks with remainders, with and without absorption, one and several
problems, and more problems than fit at once.

Bound: two FP32 evaluations that round differently.  A step rounds about thirty
times (FFT stages and updates), so 30 steps drift by some sqrt(900) unit
roundoffs of 6e-8, 2e-6 of the series; ten times that is allowed."""
import numpy as np
import pytest

import phantoms
from gpu_helpers import rel_l2, to_gpu, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EXTENTS = [24, 30, 32, 36, 40, 42, 48, 50, 54, 56, 60, 64, 70, 72, 80, 84, 90, 96, 98, 100, 108, 112, 120, 126, 128,
           140, 144, 150, 160, 168, 180, 192, 196, 200, 210, 216]
TOL = 2e-5


def contexts(shape, pml, lossless, batch, nt=30, seed=3):
    from paper_1810_11685_gb300.binding import Context
    rng = np.random.default_rng(seed + shape[0])
    full = tuple(n + 2 * pml for n in shape)
    dx = 1e-4
    c = 1500.0 + 80.0 * rng.standard_normal(full).clip(-1, 1)
    rho = 1000.0 + 50.0 * rng.standard_normal(full).clip(-1, 1)
    alpha = None if lossless else rng.uniform(0.3, 1.0, full)
    half = np.array([(shape[1] - 1) / 2 * dx, (shape[0] - 1) / 2 * dx])
    sensors = rng.uniform(-1, 1, (11, 2)) * half
    kw = dict(dx=dx, dt=0.3 * dx / c.max(), nt=nt, pml=pml, y=1.5, lossless=lossless, precision="fp32", max_batch=batch)
    return [Context(c, rho, alpha, np.full(shape, 1e-3), sensors, generic_fft=g, **kw) for g in (False, True)], rng


def check(shape, pml, lossless, batch):
    (a, g), rng = contexts(shape, pml, lossless, batch)
    p0 = to_gpu(rng.standard_normal((batch,) + shape), torch.float32)
    W = to_gpu(rng.standard_normal((batch, a.nt, a.ns)), torch.float32)
    d, dg = a.acoustic_forward(p0), g.acoustic_forward(p0)
    h, hg = a.acoustic_adjoint(W), g.acoustic_adjoint(W)
    a.sync()
    assert a.stats()["launches"] == 2                    # the loop kernel ran: one launch each
    for b in range(batch):
        assert rel_l2(to_np(d[b]), to_np(dg[b])) <= TOL
        assert rel_l2(to_np(h[b]), to_np(hg[b])) <= TOL


@pytest.mark.parametrize("lossless", [False, True])
@pytest.mark.parametrize("extent", EXTENTS)
def test_square_extents(extent, lossless):
    pml = 4 if extent < 60 else 10
    check((extent - 2 * pml,) * 2, pml, lossless, 1)


@pytest.mark.parametrize("lossless", [False, True])
@pytest.mark.parametrize("full", [(24, 30), (56, 40), (210, 24), (48, 216), (150, 210), (100, 126), (168, 120)])
def test_uneven_grids_at_runtime_lengths(full, lossless):
    check((full[0] - 8, full[1] - 8), 4, lossless, 2)


@pytest.mark.parametrize("extent,batch", [(32, 40), (96, 21), (120, 17)])
def test_many_problems(extent, batch):
    check((extent - 8,) * 2, 4, False, batch)


@pytest.mark.parametrize("lossless", [False, True])
def test_checkpoints_on_an_uneven_grid(lossless):
    (a, _), rng = contexts((52, 62), 4, lossless, 2, nt=23)
    p0 = to_gpu(rng.standard_normal((2, 52, 62)), torch.float32)
    full = a.acoustic_forward(p0)
    for K in (1, 5, 22):
        data, ck = a.acoustic_forward_ckpt(p0, K)
        assert torch.equal(data, full)
        for m in range((a.nt - 1) // K):
            out = a.acoustic_resume(ck, K, m, batch=2)
            assert torch.equal(out[:, (m + 1) * K:], full[:, (m + 1) * K:])
