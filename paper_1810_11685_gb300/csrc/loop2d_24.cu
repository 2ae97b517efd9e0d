// Whole-loop kernels of square 2D FP32 grids of extent 24, 72, 144 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(24)
QPAT_LOOP_INST(72)
QPAT_LOOP_INST(144)
}  // namespace qpat
