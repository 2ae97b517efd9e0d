// Whole-loop kernels of square 2D FP32 grids of extent 50, 108, 200 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(50)
QPAT_LOOP_INST(108)
QPAT_LOOP_INST(200)
}  // namespace qpat
