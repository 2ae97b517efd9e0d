// Whole-loop kernels of square 2D FP32 grids of extent 48, 100, 196 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(48)
QPAT_LOOP_INST(100)
QPAT_LOOP_INST(196)
}  // namespace qpat
