// Whole-loop kernels of square 2D FP32 grids of extent 60, 126, and 224 without absorption (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(60)
QPAT_LOOP_INST(126)
QPAT_LOOP_INST_LOSSLESS(224)
}  // namespace qpat
