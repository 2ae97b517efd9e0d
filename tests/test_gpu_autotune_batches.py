"""qpat_autotune's choice between the whole-loop kernel and the launched passes
holds for the batch it was given, not for the others, and the pass kernels it
reports are ones that the extent has."""
import pytest

import phantoms
from gpu_helpers import rel_l2, to_gpu, to_np
from test_gpu_loop2d import contexts

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def launches(ctx, p0):
    n = ctx.stats()["launches"]
    out = ctx.acoustic_forward(p0)
    ctx.sync()
    return ctx.stats()["launches"] - n, out


def test_tuning_a_large_batch_keeps_the_loop_kernel_for_one_problem():
    (ctx, _), rng = contexts((148, 148), 10, False, 8)     # 168^2
    p0 = to_gpu(rng.standard_normal((8, 148, 148)), torch.float32)
    one, want = launches(ctx, p0[:1])
    many, want8 = launches(ctx, p0)
    assert one == 1 and many > 1                           # eight problems take two rounds of clusters
    ctx.autotune(batch=8, steps=20)
    n, out = launches(ctx, p0[:1])
    assert n == 1 and torch.equal(out, want)
    n, out = launches(ctx, p0)
    assert rel_l2(to_np(out), to_np(want8)) <= 2e-5        # two FP32 evaluations (test_gpu_loop2d)


def test_an_extent_without_specialised_passes_reports_none():
    (ctx, _), rng = contexts((104, 104), 8, False, 2)      # 120^2
    assert ctx.autotune(batch=1, steps=20) == {"fast_rows": False, "fast_cols": False}
    p0 = to_gpu(rng.standard_normal((2, 104, 104)), torch.float32)
    assert launches(ctx, p0[:1])[0] == 1 and launches(ctx, p0)[0] == 1
