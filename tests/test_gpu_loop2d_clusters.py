"""Which cluster size the whole-loop kernel takes: more problems at once take no
longer than one of them while they fit the GPU alone on their SMs, and where the
specialised passes are faster than small clusters of many points they run.

40^2: 32 problems in clusters of four take 1.05 times one problem (in clusters of
eight, two to an SM, 2.0 times): 1.4 tells them apart."""
import statistics

import pytest

from gpu_helpers import rel_l2, to_gpu, to_np
from test_gpu_loop2d import TOL, contexts

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def run_ms(ctx, p0, n=15):
    def once():
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        ctx.acoustic_forward(p0)
        b.record()
        b.synchronize()
        return a.elapsed_time(b)
    once()
    return statistics.median(once() for _ in range(n))


def test_many_small_problems_take_the_time_of_one():
    (ctx, _), rng = contexts((32, 32), 4, False, 32, nt=120)
    p0 = to_gpu(rng.standard_normal((32, 32, 32)), torch.float32)
    assert run_ms(ctx, p0) <= 1.4 * run_ms(ctx, p0[:1])


# (shape, pml, lossless, problems, whether the loop kernel runs)
@pytest.mark.parametrize("shape,lossless,batch,loop", [((32, 32), False, 12, True), ((32, 32), False, 36, True),
                                                       ((48, 48), True, 64, True), ((160, 40), True, 24, False),
                                                       ((160, 160), True, 12, False), ((88, 88), False, 33, True)])
def test_every_cluster_size_against_the_generic_passes(shape, lossless, batch, loop):
    (a, g), rng = contexts(shape, 4, lossless, batch, nt=20)
    p0 = to_gpu(rng.standard_normal((batch,) + shape), torch.float32)
    W = to_gpu(rng.standard_normal((batch, a.nt, a.ns)), torch.float32)
    d, dg = a.acoustic_forward(p0), g.acoustic_forward(p0)
    h, hg = a.acoustic_adjoint(W), g.acoustic_adjoint(W)
    a.sync()
    assert (a.stats()["launches"] == 2) == loop
    for b in (0, batch // 2, batch - 1):
        assert rel_l2(to_np(d[b]), to_np(dg[b])) <= TOL
        assert rel_l2(to_np(h[b]), to_np(hg[b])) <= TOL
