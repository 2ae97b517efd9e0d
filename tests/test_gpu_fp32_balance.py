"""FP32 fields that share a transform although one of them is far weaker: waves
along one axis (the other velocity is near zero) and exponents near 1 and 2 and
above, where the balance factors of the absorption terms reach their limits, in
the whole-loop kernel, the specialised and the generic passes, against the FP64
context on the same inputs.

Bound: a step rounds about thirty times (FFT stages and updates) by the unit
roundoff 6e-8; sixty steps drift by some sqrt(1800) of them, 2.5e-6 of the series;
ten times that is allowed."""
import numpy as np
import pytest

from gpu_helpers import rel_l2, to_gpu, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL, NT, DX = 2.5e-5, 60, 1e-4


def context(shape, pml, y, axis, precision, generic):
    from paper_1810_11685_gb300.binding import Context
    full = tuple(n + 2 * pml for n in shape)
    t = np.linspace(-0.8, 0.8, 24)
    line = np.stack([t, 0.1 + 0 * t], 1)[:, ::-1 if axis else 1] * (np.array(shape[::-1]) - 1) / 2 * DX
    return Context(np.full(full, 1500.0), np.full(full, 1000.0), np.full(full, 0.75), np.full(shape, 1e-3), line, dx=DX,
                   dt=0.3 * DX / 1500, nt=NT, pml=pml, y=y, precision=precision, generic_fft=generic)


# 96^2, 70 x 84: loop kernel; 288^2: specialised passes; 96^2 generic: generic passes
@pytest.mark.parametrize("shape,pml,generic", [((80, 80), 8, False), ((54, 68), 8, False), ((256, 256), 16, False),
                                               ((80, 80), 8, True)])
@pytest.mark.parametrize("y", [1.02, 1.5, 1.98, 2.02, 2.5])
@pytest.mark.parametrize("axis", [0, 1])
def test_wave_along_one_axis(shape, pml, generic, y, axis):
    X = np.arange(shape[axis]).reshape((-1, 1) if axis == 0 else (1, -1)) - shape[axis] / 2
    T = np.arange(shape[1 - axis]).reshape((1, -1) if axis == 0 else (-1, 1)) + 0.5
    p0 = (np.exp(-(X / 5.0) ** 2) * np.sin(np.pi * T / shape[1 - axis]) ** 2).astype(np.float32)
    W = np.sin(0.2 * np.arange(NT))[:, None].astype(np.float32) * np.ones((1, 24), np.float32)
    lo, hi = (context(shape, pml, y, axis, p, generic) for p in ("fp32", "fp64"))
    got = to_np(lo.acoustic_forward(to_gpu(p0, torch.float32))), to_np(lo.acoustic_adjoint(to_gpu(W, torch.float32)))
    ref = to_np(hi.acoustic_forward(to_gpu(p0, torch.float64))), to_np(hi.acoustic_adjoint(to_gpu(W, torch.float64)))
    lo.sync()
    hi.sync()
    for a, b in zip(got, ref):
        assert rel_l2(a, b) <= TOL
