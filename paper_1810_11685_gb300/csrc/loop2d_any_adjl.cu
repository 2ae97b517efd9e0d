// Whole-loop kernel of 2D FP32 grids at runtime lengths (see loop2d.cuh): H_a^*, lossless.
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST0(true, true)
}  // namespace qpat
