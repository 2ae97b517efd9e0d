"""A refused launch of the whole-loop kernel is reported, by every call that
runs it and every time: the library is linked with a stand-in for the host side
of that kernel whose launches come back as cudaErrorInvalidConfiguration."""
import ctypes
import glob
import os
import subprocess

import pytest

import phantoms
from gpu_helpers import rel_l2, to_gpu, to_np

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ECUDA = 7

STANDIN = r"""
#include "loop2d.h"
namespace qpat {
void loop_plan(const PropArgs<float>&, int, int, LoopPlan* p) {
  *p = LoopPlan{};
  p->ok = p->own_kernel = 1;
}
int loop_waves(const LoopPlan&, int) { return 1; }
cudaError_t launch_loop(const PropArgs<float>&, const LoopPlan&, int, int, int, int, int, int, int, int, int, int,
                        cudaStream_t) {
  return cudaErrorInvalidConfiguration;
}
}  // namespace qpat
"""


@pytest.fixture(scope="module")
def refusing(tmp_path_factory):
    from paper_1810_11685_gb300 import binding, build
    build.build()
    d = tmp_path_factory.mktemp("standin")
    src, lib = d / "loop2d.cu", d / "libqpat_standin.so"
    src.write_text(STANDIN)
    objs = [o for o in glob.glob(os.path.join(build.BUILD, "*.o"))
            if not os.path.basename(o).startswith("loop2d")
            and os.path.exists(os.path.join(build.CSRC, os.path.basename(o)[:-2] + ".cu"))]
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-o", str(lib), str(src), *objs], check=True)
    keep = binding._lib, binding._LIB_PATH
    binding._lib, binding._LIB_PATH = None, str(lib)
    yield binding
    binding._lib, binding._LIB_PATH = keep


def test_every_call_reports_it(refusing):
    w = phantoms.small(n=40, pml=8, nt=12, n_sensors=6, seed=2)
    for no_graphs in (False, True):
        ctx = refusing.context_from_workload(w, precision="fp32", max_batch=2, no_graphs=no_graphs)
        p0 = to_gpu(phantoms.smooth_p0(w), torch.float32)[None]
        W = to_gpu(phantoms.random_field((1, w.nt, w.n_sensors), 1), torch.float32)
        group = refusing.Group([ctx])
        calls = [lambda: ctx.acoustic_forward(p0), lambda: ctx.acoustic_adjoint(W),
                 lambda: ctx.acoustic_forward_ckpt(p0, 3), lambda: group.acoustic_forward([p0]),
                 lambda: group.acoustic_adjoint([W]), lambda: group.tune([1], steps=4)]
        for call in calls:
            for _ in range(2):                                 # nothing without the kernel is kept for the next call
                with pytest.raises(refusing.QpatError) as e:
                    call()
                assert e.value.status == ECUDA
        # the launched passes are not touched by it, and the tuner keeps them
        ctx.profile("F_R1")
        want = ctx.acoustic_forward(p0)
        ctx.profile(None)
        ctx.autotune(batch=1, steps=4)
        assert rel_l2(to_np(ctx.acoustic_forward(p0)), to_np(want)) <= 2e-5
        ctx.sync()
        group.close()
        ctx.close()
