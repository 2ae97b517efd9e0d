"""Checkpoints of small 2D FP32 grids resumed by other kernels than those that
stored them: the whole-loop kernel's by the launched passes and the other way
round, on the same context (profiled calls and other batches run other kernels)
and on a generic_fft context of the same grid.

Bound: two FP32 evaluations that round differently.  A step rounds about thirty
times (FFT stages and updates), so 23 steps drift by some sqrt(700) unit
roundoffs of 6e-8, 1.6e-6 of the series; ten times that and a little is allowed."""
import numpy as np
import pytest

from gpu_helpers import rel_l2, to_gpu, to_np
from test_gpu_loop2d import contexts

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 2e-5
NT = 23


def setup(shape, lossless, batch):
    (loop, generic), rng = contexts(shape, 4, lossless, batch, nt=NT)
    return loop, generic, to_gpu(rng.standard_normal((batch,) + shape), torch.float32)


def resumed(ctx, ck, K, m, batch, data, exact):
    out = ctx.acoustic_resume(ck, K, m, batch=batch)[:, (m + 1) * K:]
    want = data[:batch, (m + 1) * K:]
    ctx.sync()
    if exact:
        assert torch.equal(out, want)
    else:
        assert rel_l2(to_np(out), to_np(want)) <= TOL


@pytest.mark.parametrize("lossless", [False, True])
@pytest.mark.parametrize("shape", [(88, 88), (52, 62)])
@pytest.mark.parametrize("K", [1, 5, 22])
def test_loop_kernel_and_launched_passes(shape, lossless, K):
    loop, generic, p0 = setup(shape, lossless, 2)
    data, ck = loop.acoustic_forward_ckpt(p0, K)
    gdata, gck = generic.acoustic_forward_ckpt(p0, K)
    loop.profile("F_R2")                                   # profiled calls run the launched passes
    pdata, pck = loop.acoustic_forward_ckpt(p0, K)
    for m in range((NT - 1) // K):
        resumed(loop, ck, K, m, 2, data, False)
        resumed(loop, pck, K, m, 2, pdata, True)
    loop.profile(None)
    for m in range((NT - 1) // K):
        resumed(loop, ck, K, m, 2, data, True)
        resumed(loop, pck, K, m, 2, pdata, False)
        resumed(loop, gck, K, m, 2, gdata, False)
        resumed(generic, ck, K, m, 2, data, False)


@pytest.mark.parametrize("lossless", [False, True])
def test_first_checkpoint_at_a_smaller_batch(lossless):
    """168^2: eight problems run the launched passes, one the loop kernel."""
    loop, _, p0 = setup((160, 160), lossless, 8)
    data, ck = loop.acoustic_forward_ckpt(p0, 5)
    resumed(loop, ck, 5, 0, 1, data, False)
    resumed(loop, ck, 5, 3, 8, data, True)


def test_resume_after_autotune():
    loop, _, p0 = setup((52, 62), False, 2)
    data, ck = loop.acoustic_forward_ckpt(p0, 5)
    loop.autotune(batch=2, steps=8)
    resumed(loop, ck, 5, 1, 2, data, False)
