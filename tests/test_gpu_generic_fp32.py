"""The generic FP32 passes at extents whose runtime Stockham plans have the
radices that only FP32 uses, 6 and 9, alone and repeated, against the FP64 oracle
(FP64 plans hold 2, 3, 4, 5, 7 and 8).

Bound: a step rounds about thirty times (FFT stages and updates) by the unit
roundoff 6e-8; twelve steps drift by some sqrt(360) of them, 1.2e-6 of the series;
ten times that is allowed."""
import numpy as np
import pytest

import phantoms
from oracle import acoustic
from gpu_helpers import make_pair, rel_l2, to_gpu, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1.2e-5


# 12 = 4 3, 18 = 6 3, 24 = 8 3, 36 = 4 9, 42 = 6 7, 54 = 6 9, 90 = 6 3 5, 108 = 4 9 3, 162 = 6 9 3, 324 = 4 9 9, 486 = 6 9 9
@pytest.mark.parametrize("extent", [12, 18, 24, 36, 42, 54, 90, 108, 162, 324, 486])
@pytest.mark.parametrize("batch", [1, 7])
def test_every_radix_fp32(extent, batch):
    pml = 2 if extent < 24 else 4
    w = phantoms.small(n=extent - 2 * pml, pml=pml, nt=12, n_sensors=6, seed=extent)
    ctx, S = make_pair(w, "fp32", max_batch=batch, generic_fft=True)
    p0 = np.stack([phantoms.random_field(w.interior_shape, 3 + b) for b in range(batch)]).astype(np.float32)
    W = np.stack([phantoms.random_field((w.nt, w.n_sensors), 40 + b) for b in range(batch)]).astype(np.float32)
    data = to_np(ctx.acoustic_forward(to_gpu(p0, torch.float32)))
    adj = to_np(ctx.acoustic_adjoint(to_gpu(W, torch.float32)))
    ctx.sync()
    for b in (0, batch - 1):
        assert rel_l2(data[b], acoustic.forward(S, p0[b].astype(np.float64))) <= TOL
        assert rel_l2(adj[b], acoustic.adjoint(S, W[b].astype(np.float64))) <= TOL
