// Whole-loop kernels of square 2D FP32 grids of extent 40, 96, 180 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(40)
QPAT_LOOP_INST(96)
QPAT_LOOP_INST(180)
}  // namespace qpat
