// Whole-loop kernels of square 2D FP32 grids of extent 42, 98, 192 (see loop2d.cuh).
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST(42)
QPAT_LOOP_INST(98)
QPAT_LOOP_INST(192)
}  // namespace qpat
