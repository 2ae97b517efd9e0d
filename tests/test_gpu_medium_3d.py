"""The medium derivatives need a 2D context: on a 3D one of either precision
both calls come back as EINVAL, and the context stays usable."""
import numpy as np
import pytest

import phantoms
from gpu_helpers import to_gpu

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

EINVAL = 1


@pytest.mark.parametrize("lossless", [False, True])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_3d_contexts_are_refused(prec, lossless):
    from paper_1810_11685_gb300.binding import Context, QpatError
    n, pml, dx = 8, 4, 1e-4
    full = (n + 2 * pml,) * 3
    sensors = np.zeros((2, 3))
    sensors[1] = dx
    ctx = Context(np.full(full, 1500.0), np.full(full, 1000.0), None if lossless else np.full(full, 0.7),
                  np.full((n,) * 3, 1e-3 / 3), sensors, dx=dx, dt=0.2 * dx / 1500, nt=5, pml=pml, y=1.5,
                  lossless=lossless, precision=prec)
    p0 = to_gpu(phantoms.random_field((n,) * 3, 1), torch.float64)
    w = torch.ones(ctx.nt, ctx.ns, dtype=torch.float64, device="cuda")
    for call in (lambda: ctx.vjp_medium(p0, w), lambda: ctx.jvp_medium(p0)):
        with pytest.raises(QpatError) as e:
            call()
        assert e.value.status == EINVAL
    ctx.acoustic_forward(p0.to(ctx.dtype))
    ctx.sync()
