// Whole-loop kernels of square 2D FP32 grids of extent 54, 112, 210 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(54)
QPAT_LOOP_INST(112)
QPAT_LOOP_INST(210)
}  // namespace qpat
