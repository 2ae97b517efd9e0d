// Whole-loop kernels of square 2D FP32 grids of extent 60, 126, 224 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(60)
QPAT_LOOP_INST(126)
QPAT_LOOP_INST(224)
}  // namespace qpat
