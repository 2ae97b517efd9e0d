// Whole-loop kernels of square 2D FP32 grids of extent 56, 120, 216 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(56)
QPAT_LOOP_INST(120)
QPAT_LOOP_INST(216)
}  // namespace qpat
