// Host side of the whole-loop kernel (loop2d.cuh): radices, fit and launch.
#include <map>
#include <mutex>
#include <tuple>

#include "loop2d.h"

namespace qpat {

namespace {
int line_stride(const LoopAxis& x, const LoopAxis& y) {
  const int a = loop_line(x), b = loop_line(y);
  return (a > b ? a : b) | 1;                                    // odd: adjacent lines start on other banks
}
int ceil_div(int a, int b) { return (a + b - 1) / b; }
constexpr int kClusters[3] = {16, 8, 4};
}  // namespace

size_t loop_smem(const PropArgs<float>& a, const LoopAxis& x, const LoopAxis& y, int nc, int adj, int lossless) {
  return loop_layout(x, y, ceil_div(a.ny / 2, nc), ceil_div(a.nxh, nc), line_stride(x, y), adj != 0, lossless != 0)
             .total *
         sizeof(float);
}

namespace {
// Extent of a grid's kernels: its own where square grids of it have some, 0
// (runtime lengths) otherwise.
int kernel_extent(const PropArgs<float>& a) {
  if (a.nx != a.ny) return 0;
  switch (a.nx) {
#define QPAT_LOOP_CASE(L) case L: return L;
    QPAT_LOOP_EXTENTS(QPAT_LOOP_CASE)
#undef QPAT_LOOP_CASE
    default: return 0;
  }
}
int occupancy_query(int L, int adj, int ll, int nc, size_t smem) {
  switch (L) {
#define QPAT_LOOP_CASE(L) case L: return loop_occupancy_len<L>(adj, ll, nc, smem);
    QPAT_LOOP_EXTENTS(QPAT_LOOP_CASE)
#undef QPAT_LOOP_CASE
    default: return 0;
  }
}
// The query takes about a millisecond, a context creation several; its answer
// depends on nothing but the arguments and the device.
int occupancy(int L, int adj, int ll, int nc, size_t smem) {
  static std::mutex mtx;
  static std::map<std::tuple<int, int, int, int, int, size_t>, int> known;
  int dev = 0;
  cudaGetDevice(&dev);
  const std::tuple<int, int, int, int, int, size_t> key(dev, L, adj, ll, nc, smem);
  std::lock_guard<std::mutex> lock(mtx);
  const auto it = known.find(key);
  if (it != known.end()) return it->second;
  const int n = occupancy_query(L, adj, ll, nc, smem);
  if (n > 0) known[key] = n;
  return n;
}
}  // namespace

void loop_plan(const PropArgs<float>& a, int lossless, int max_batch, LoopPlan* p) {
  *p = LoopPlan{};
  p->x = loop_axis(a.nx);
  p->y = loop_axis(a.ny);
  if (!p->x.L || !p->y.L) return;
  const int L = kernel_extent(a);
  p->own_kernel = L != 0;
  // the adjoint kernel holds more than the forward one: it decides the fit
  // (smaller clusters are only looked at when max_batch may not fit as 16s)
  if (!occupancy(L, 0, lossless, 0, 0)) return;
  for (int k = 0; k < 3; ++k) {
    p->max_clusters[k] = occupancy(L, 1, lossless, kClusters[k], loop_smem(a, p->x, p->y, kClusters[k], 1, lossless));
    p->ok = p->ok || p->max_clusters[k] > 0;
    if (k == 0 && p->max_clusters[0] >= max_batch) break;
  }
}

namespace {
// Cluster size (index into kClusters) for `batch` problems: the fewest rounds
// of resident clusters, weighted by the time of a step (96^2: 16 CTAs 14.6 us,
// 8 16.7 us, 4 23.4 us); 16 for one round.
int choose(const LoopPlan& p, int batch) {
  static const double cost[3] = {1.0, 1.15, 1.6};
  int k = -1;
  double best = 1e300;
  for (int q = 0; q < 3; ++q) {
    if (p.max_clusters[q] <= 0) continue;
    const double c = cost[q] * ceil_div(batch, p.max_clusters[q]);
    if (c < best) { best = c; k = q; }
  }
  return k;
}
}  // namespace

int loop_waves(const LoopPlan& p, int batch) {
  const int k = choose(p, batch);
  return k < 0 ? 1 << 30 : ceil_div(batch, p.max_clusters[k]);
}

cudaError_t launch_loop(const PropArgs<float>& a, const LoopPlan& p, int adj, int lossless, int batch, int nt, int g0,
                        int g1, int load, int save, int rebuild, int gather_last, cudaStream_t s) {
  const int k = choose(p, batch);
  if (k < 0) return cudaErrorInvalidConfiguration;
  const int nc = kClusters[k];
  LoopArgs A{};
  A.a = a;
  A.x = p.x;
  A.y = p.y;
  A.rp = ceil_div(a.ny / 2, nc);
  A.cp = ceil_div(a.nxh, nc);
  A.stride = line_stride(p.x, p.y);
  A.nt = nt;
  A.g0 = g0;
  A.g1 = g1;
  A.load = load;
  A.save = save;
  A.rebuild = rebuild;
  A.gather_last = gather_last;
  const size_t smem = loop_smem(a, p.x, p.y, nc, adj, lossless);
  switch (kernel_extent(a)) {
#define QPAT_LOOP_CASE(L) case L: return loop_launch_len<L>(A, adj, lossless, nc, batch, smem, s);
    QPAT_LOOP_EXTENTS(QPAT_LOOP_CASE)
#undef QPAT_LOOP_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace qpat
