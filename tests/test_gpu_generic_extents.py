"""The generic passes at extents that exercise every radix of the runtime
Stockham plan and every column width, against the FP64 oracle.

The bound is the one of the other FP64 parity tests (relative L2 1e-10: about
ten FFT stages and updates per step, each of unit roundoff 1.1e-16, over a few
dozen steps, stay below 1e-12)."""
import numpy as np
import pytest

import phantoms
from oracle import acoustic
from gpu_helpers import make_pair, rel_l2, to_gpu, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# FFT extents: 8, 10 = 2 5, 18 = 6 3, 24 = 8 3, 36 = 4 9, 42 = 6 7, 54 = 6 9, 90 = 6 3 5, 144 = 8 6 3, 162 = 6 9 3
@pytest.mark.parametrize("extent", [8, 10, 18, 24, 36, 42, 54, 90, 144, 162])
@pytest.mark.parametrize("batch", [1, 7])
def test_every_radix_fp64(extent, batch):
    pml = 2 if extent < 24 else 4
    w = phantoms.small(n=extent - 2 * pml, pml=pml, nt=12, n_sensors=6, seed=extent)
    ctx, S = make_pair(w, "fp64", max_batch=batch)
    p0 = np.stack([phantoms.random_field(w.interior_shape, 3 + b) for b in range(batch)])
    W = np.stack([phantoms.random_field((w.nt, w.n_sensors), 40 + b) for b in range(batch)])
    data = to_np(ctx.acoustic_forward(to_gpu(p0, torch.float64)))
    adj = to_np(ctx.acoustic_adjoint(to_gpu(W, torch.float64)))
    ctx.sync()
    for b in (0, batch - 1):
        assert rel_l2(data[b], acoustic.forward(S, p0[b])) <= 1e-10
        assert rel_l2(adj[b], acoustic.adjoint(S, W[b])) <= 1e-10
