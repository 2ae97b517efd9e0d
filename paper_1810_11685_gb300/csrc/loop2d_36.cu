// Whole-loop kernels of square 2D FP32 grids of extent 36, 90, 168 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(36)
QPAT_LOOP_INST(90)
QPAT_LOOP_INST(168)
}  // namespace qpat
