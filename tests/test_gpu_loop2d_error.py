"""The whole-loop kernel is no further from the FP64 fields than the launched
passes at the extents where its radices once made the rounding of the DFT
constants add up (60, 108, 180, 192, 216 and uneven grids with them).

Both kinds of passes have the same number of roundings a step; which constants a
length uses makes their errors differ by up to 1.1 in the launched passes alone
(240^2 to 1080^2, several radix plans).  So: at most 1.1 times theirs."""
import numpy as np
import pytest

from gpu_helpers import rel_l2, to_gpu, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NT, DX = 150, 1e-4


def errors(shape, pml, lossless):
    from paper_1810_11685_gb300.binding import Context
    rng = np.random.default_rng(5 + shape[0])
    full = tuple(n + 2 * pml for n in shape)
    y, x = np.mgrid[0:full[0], 0:full[1]]
    c = 1500.0 + 60.0 * np.sin(2 * np.pi * (2 * x / full[1] + y / full[0]) + 1.0)
    rho = 1000.0 + 60.0 * np.cos(2 * np.pi * (x / full[1] - 2 * y / full[0]))
    th = 2 * np.pi * np.arange(48) / 48
    sensors = 0.9 * np.stack([np.cos(th) * (shape[1] - 1), np.sin(th) * (shape[0] - 1)], 1) / 2 * DX
    p0 = rng.standard_normal((1,) + shape).astype(np.float32)
    W = rng.standard_normal((1, NT, 48)).astype(np.float32)
    out = {}
    for name, prec, generic in (("exact", "fp64", False), ("loop", "fp32", False), ("passes", "fp32", True)):
        ctx = Context(c, rho, None if lossless else np.full(full, 0.75), np.full(shape, 5e-4), sensors, dx=DX,
                      dt=0.3 * DX / c.max(), nt=NT, pml=pml, y=1.5, lossless=lossless, precision=prec,
                      generic_fft=generic)
        out[name] = [to_np(ctx.acoustic_forward(to_gpu(p0, ctx.dtype))),
                     to_np(ctx.acoustic_adjoint(to_gpu(W, ctx.dtype)))]
        ctx.sync()
        ctx.close()
    return [[rel_l2(a, e) for a, e in zip(out[k], out["exact"])] for k in ("loop", "passes")]


@pytest.mark.parametrize("lossless", [False, True])
@pytest.mark.parametrize("full", [(60, 60), (108, 108), (180, 180), (192, 192), (216, 216), (60, 90), (216, 48)])
def test_error_against_fp64(full, lossless):
    loop, passes = errors((full[0] - 20, full[1] - 20), 10, lossless)
    for a, b in zip(loop, passes):
        assert a <= 1.1 * b
