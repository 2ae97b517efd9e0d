"""Groups whose shape was never set: members that each fill the GPU run in turn,
others as branches; either way each member has the bits of its own calls."""
import dataclasses

import pytest

import phantoms
from gpu_helpers import make_pair, to_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 288^2 x 13 and 432^2 x 6 are each above a million points, 288^2 x 12 and 432^2 x 5 below
@pytest.mark.parametrize("batches", [(13, 6), (12, 6), (13, 5), (13, 0)])
def test_unset_shape_equals_individual_calls(batches):
    from paper_1810_11685_gb300.binding import Group
    ws = [dataclasses.replace(w, nt=nt) for w, nt in zip(phantoms.c4_workloads()[:2], (5, 7))]
    ctxs = [make_pair(w, "fp32", max_batch=13)[0] for w in ws]
    g = Group(ctxs)
    p0s = [to_gpu(phantoms.random_field((b,) + w.interior_shape, 3), torch.float32) if b else None
           for w, b in zip(ws, batches)]
    Ws = [to_gpu(phantoms.random_field((b, w.nt, w.n_sensors), 4), torch.float32) if b else None
          for w, b in zip(ws, batches)]
    for outs, own, ins in ((g.acoustic_forward(p0s), "acoustic_forward", p0s),
                           (g.acoustic_adjoint(Ws), "acoustic_adjoint", Ws)):
        for c, o, x in zip(ctxs, outs, ins):
            assert (o is None) if x is None else torch.equal(o, getattr(c, own)(x))
    g.close()
