// Whole-loop kernels of square 2D FP32 grids of extent 32, 84, 160 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(32)
QPAT_LOOP_INST(84)
QPAT_LOOP_INST(160)
}  // namespace qpat
