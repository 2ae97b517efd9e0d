// Whole-loop kernel of 2D FP32 grids at runtime lengths (see loop2d.cuh): H_a with absorption.
#include "loop2d.cuh"
namespace qpat {
extern template int loop_occupancy_one<false, true, 0>(int, size_t);
extern template int loop_occupancy_one<true, false, 0>(int, size_t);
extern template int loop_occupancy_one<true, true, 0>(int, size_t);
extern template cudaError_t loop_launch_one<false, true, 0>(const LoopArgs&, int, int, size_t, cudaStream_t);
extern template cudaError_t loop_launch_one<true, false, 0>(const LoopArgs&, int, int, size_t, cudaStream_t);
extern template cudaError_t loop_launch_one<true, true, 0>(const LoopArgs&, int, int, size_t, cudaStream_t);
QPAT_LOOP_INST0(false, false)

template <>
cudaError_t loop_launch_len<0>(const LoopArgs& A, int adj, int ll, int nc, int batch, size_t smem, cudaStream_t s) {
  if (adj) return ll ? loop_launch_one<true, true, 0>(A, nc, batch, smem, s) : loop_launch_one<true, false, 0>(A, nc, batch, smem, s);
  return ll ? loop_launch_one<false, true, 0>(A, nc, batch, smem, s) : loop_launch_one<false, false, 0>(A, nc, batch, smem, s);
}
template <>
int loop_occupancy_len<0>(int adj, int ll, int nc, size_t smem) {
  if (adj) return ll ? loop_occupancy_one<true, true, 0>(nc, smem) : loop_occupancy_one<true, false, 0>(nc, smem);
  return ll ? loop_occupancy_one<false, true, 0>(nc, smem) : loop_occupancy_one<false, false, 0>(nc, smem);
}
}  // namespace qpat
