// Whole-loop kernels of square 2D FP32 grids of extent 70, 140 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(70)
QPAT_LOOP_INST(140)
}  // namespace qpat
