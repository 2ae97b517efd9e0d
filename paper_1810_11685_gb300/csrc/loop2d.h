// Whole time loops of small 2D FP32 grids in one launch: a thread-block
// cluster per problem runs every pass of H_a or H_a^* (loop2d.cuh).
#pragma once
#include "qpat_internal.h"

namespace qpat {

// Threads per CTA of the kernel of extent L (0: runtime lengths): about one
// butterfly of a stage each.
constexpr int loop_threads(int L) { return L == 0 || L > 168 ? 384 : 256; }
constexpr int kLoopMaxCluster = 16;

// Radices of one axis, L = q[0] q[1] q[2]; L = 0: none.
struct LoopAxis {
  int L;
  int q[3];
};
// q0 in 3..8, q1 in 2..8, q2 in 4..8, by the instructions of one radix-R
// butterfly of a packed pair with its index arithmetic (counted from the
// source; only their order matters).  Of equal plans one with 3 in the middle, where
// q2 is at most 5: 60 as 5 3 4 instead of 3 5 4 has 0.87 of the error against 64 bits
// and takes 0.98 of the time, 48 0.92 and 0.99, 72 0.99 and 0.98 (108 as 6 3 6 1.02
// and 1.02).
constexpr LoopAxis loop_axis(int L) {
  const int cost[9] = {0, 0, 30, 45, 55, 85, 100, 150, 130};
  LoopAxis ax{0, {0, 0, 0}};
  int best = 1 << 30;
  for (int r = 4; r <= 8; ++r)
    for (int p = 3; p <= 8; ++p) {
      if (L % (p * r)) continue;
      const int m = L / (p * r);
      if (m < 2 || m > 8) continue;
      const int c = cost[p] + cost[r] + cost[m];
      if (c < best || (c == best && m == 3 && ax.q[1] != 3 && r <= 5)) {
        best = c;
        ax = LoopAxis{L, {p, m, r}};
      }
    }
  return ax;
}
// Plane pitch of a first stage of nb butterflies: butterfly j leaves output r
// at r pitch + j, 5 mod 8 so that a warp reading the next stage's operands
// (planes cycling fastest) spreads over the banks.
__host__ __device__ constexpr int loop_pitch(int nb) { return nb + ((5 - nb) % 8 + 8) % 8; }
// 16-byte entries of one line: either first stage's planes or the line itself.
__host__ __device__ constexpr int loop_line(const LoopAxis& a) {
  const int x = a.q[0] * loop_pitch(a.L / a.q[0]), y = a.q[2] * loop_pitch(a.L / a.q[2]);
  return x > y ? x : y;
}
// Twiddles of one axis, stage by stage (LoopTw): mid and last of both orders.
__host__ __device__ constexpr int loop_ntw(const LoopAxis& a) {
  return a.q[0] * (a.q[1] - 1) + a.q[0] * a.q[1] * (a.q[2] - 1) + a.q[2] * (a.q[1] - 1) +
         a.q[2] * a.q[1] * (a.q[0] - 1);
}

struct LoopPlan {
  int ok = 0;              // the grid has a plan and one problem fits a cluster
  int own_kernel = 0;      // square grid of an extent with compile-time kernels
  LoopAxis x{}, y{};
  bool specialised = false;  // the launched passes are specialised on both axes
  double shared_cost = 1.0;  // time of a round with two CTAs to an SM against one with one
  int alone[3] = {0, 0, 0};  // clusters of 16, 8, 4 CTAs resident with one CTA to an SM (0: does not fit)
  int max_clusters[3] = {0, 0, 0}; // clusters resident at once
};

struct LoopArgs {
  PropArgs<float> a;
  LoopAxis x, y;
  int rp, cp;              // row pairs, column pairs per CTA
  int stride;              // 16-byte entries per line of the Stockham buffers
  int nt;                  // samples of the loop
  int g0, g1;              // passes [g0, g1) of the loop (loop_pass)
  int load, save;          // restore the state from / leave it in the context's arrays
  int rebuild;             // pass g0 only forms the pressure's spectrum from the restored state (F_R3L)
  int gather_last;         // gather sample nt - 1 at the end (forward)
};

// Shared-memory layout of one CTA in floats (every block a multiple of 16 bytes).
struct LoopLayout {
  size_t tw, fields, ktab, pml, total;
  int nfields, ntab, ntw;
};
__host__ __device__ inline size_t loop_r4(size_t n) { return (n + 3) & ~(size_t)3; }
__host__ __device__ inline LoopLayout loop_layout(const LoopAxis& x, const LoopAxis& y, int rp, int cp, int stride,
                                                  bool adj, bool ll) {
  LoopLayout l;
  l.nfields = (adj ? (ll ? 5 : 6) : 4) + (ll ? 4 : 6);
  l.ntab = ll ? 1 : 3;
  l.ntw = loop_ntw(x) + loop_ntw(y);
  l.tw = (size_t)2 * (rp > cp ? rp : cp) * stride * 4;
  l.fields = l.tw + loop_r4(2 * (size_t)(l.ntw + 2 * y.L));
  l.ktab = l.fields + loop_r4((size_t)l.nfields * rp * x.L * 2);
  l.pml = l.ktab + loop_r4((size_t)l.ntab * cp * y.L);
  l.total = l.pml + loop_r4(2 * (size_t)x.L + 4 * (size_t)rp);
  return l;
}
// Extents with kernels of their own (square grids; 224 without absorption only); the others, and uneven
// grids, run the kernels for runtime lengths.  (Both on the same square grid, one
// problem, 200 steps, forward + adjoint, runtime / compile-time length, ms: 56^2
// 9.19 / 5.71, 96^2 8.96 / 5.81, 120^2 10.1 / 6.34, 168^2 12.2 / 8.78, 210^2
// 14.7 / 11.3.)
#define QPAT_LOOP_EXTENTS(X) \
  X(24) X(30) X(32) X(36) X(40) X(42) X(48) X(50) X(54) X(56) X(60) X(64) \
  X(70) X(72) X(80) X(84) X(90) X(96) X(98) X(100) X(108) X(112) X(120) X(126) \
  X(128) X(140) X(144) X(150) X(160) X(168) X(180) X(192) X(196) X(200) X(210) X(216) \
  X(224) \
  X(0)

// Shared memory of one CTA of the loop kernel.
size_t loop_smem(const PropArgs<float>& a, const LoopAxis& x, const LoopAxis& y, int nc, int adj, int lossless);
// Plan of a grid; sets the kernels' attributes.
void loop_plan(const PropArgs<float>& a, int lossless, int max_batch, LoopPlan* p);
// Rounds of resident clusters that `batch` problems take; more than any
// number where the launched passes are known to be faster.
int loop_waves(const LoopPlan& p, int batch);
// Passes [g0, g1) of H_a (adj = 0) or H_a^* (adj = 1) of nt samples for
// `batch` problems.
cudaError_t launch_loop(const PropArgs<float>& a, const LoopPlan& p, int adj, int lossless, int batch, int nt, int g0,
                        int g1, int load, int save, int rebuild, int gather_last, cudaStream_t s);
// Per extent L (0: runtime lengths), instantiated in loop2d_*.cu.
template <bool ADJ, bool LL, int L>
cudaError_t loop_launch_one(const LoopArgs& A, int nc, int batch, size_t smem, cudaStream_t s);
template <bool ADJ, bool LL, int L>
int loop_occupancy_one(int nc, size_t smem);
template <int L>
cudaError_t loop_launch_len(const LoopArgs& A, int adj, int lossless, int nc, int batch, size_t smem, cudaStream_t s);
template <int L>
int loop_occupancy_len(int adj, int lossless, int nc, size_t smem);

}  // namespace qpat
