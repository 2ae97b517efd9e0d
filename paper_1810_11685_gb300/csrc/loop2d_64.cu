// Whole-loop kernels of square 2D FP32 grids of extent 64, 128 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(64)
QPAT_LOOP_INST(128)
}  // namespace qpat
