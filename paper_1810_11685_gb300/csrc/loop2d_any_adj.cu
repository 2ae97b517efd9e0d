// Whole-loop kernel of 2D FP32 grids at runtime lengths (see loop2d.cuh): H_a^* with absorption.
#include "loop2d.cuh"
namespace qpat {
QPAT_LOOP_INST0(true, false)
}  // namespace qpat
