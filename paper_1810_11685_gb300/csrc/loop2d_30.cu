// Whole-loop kernels of square 2D FP32 grids of extent 30, 80, 150 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(30)
QPAT_LOOP_INST(80)
QPAT_LOOP_INST(150)
}  // namespace qpat
