"""The largest extent with a whole-loop kernel: 224^2 runs it without absorption
and, since the data would not fit, the launched passes with it; both against the
generic passes (bound of test_gpu_loop2d)."""
import pytest

from gpu_helpers import rel_l2, to_gpu, to_np
from test_gpu_loop2d import TOL, check, contexts

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_without_absorption():
    check((204, 204), 10, True, 1)


def test_with_absorption():
    (a, g), rng = contexts((204, 204), 10, False, 1)
    p0 = to_gpu(rng.standard_normal((1, 204, 204)), torch.float32)
    W = to_gpu(rng.standard_normal((1, a.nt, a.ns)), torch.float32)
    assert rel_l2(to_np(a.acoustic_forward(p0)), to_np(g.acoustic_forward(p0))) <= TOL
    assert rel_l2(to_np(a.acoustic_adjoint(W)), to_np(g.acoustic_adjoint(W))) <= TOL
    a.sync()
    assert a.stats()["launches"] > 2 * a.nt                # a launch per pass
