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
constexpr size_t kMaxSmem = 227 * 1024;
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
  p->specialised = a.fast_rows && a.fast_cols;
  bool two_power = true;
  for (const LoopAxis* x : {&p->x, &p->y})
    for (int q : x->q) two_power = two_power && (q == 2 || q == 4 || q == 8);
  p->shared_cost = !p->specialised && (lossless || two_power) ? 1.1 : 1.5;
  // (also sets both kernels' attributes; the adjoint kernel holds more than the
  // forward one and decides the fit)
  if (!occupancy(L, 0, lossless, 0, 0) || !occupancy(L, 1, lossless, 0, 0)) return;
  for (int k = 0; k < 3; ++k) {
    const size_t smem = loop_smem(a, p->x, p->y, kClusters[k], 1, lossless);
    if (smem > kMaxSmem) break;                                  // (smaller clusters need more)
    p->alone[k] = occupancy(L, 1, lossless, kClusters[k], kMaxSmem);
    p->ok = p->ok || p->alone[k] > 0;
    if (p->alone[k] >= max_batch && k == 0) {                    // no more looked up than max_batch may need
      p->max_clusters[k] = p->alone[k];
      break;
    }
    p->max_clusters[k] = occupancy(L, 1, lossless, kClusters[k], smem);
  }
}

namespace {
double points_per_cta(const LoopPlan& p, int k) { return (double)p.x.L * p.y.L / kClusters[k]; }
// Cluster size (index into kClusters) for `batch` problems, by the time of a
// step: the passes' latency and the points of a CTA, times the rounds of resident
// clusters.  A round in which two CTAs share an SM measured 1.5 rounds with
// absorption, 1.0 to 1.16 without or with radices 2, 4 and 8 only (54^2 and 56^2
// without: 1.5, so grids with specialised passes, whose smaller clusters cost
// nothing, always count 1.5).  24 steps, forward + adjoint, clusters of 16 / 8 / 4,
// ms; alone on the SMs are 7, 15 and 36 clusters: 40^2, one problem 0.67 / 0.67 /
// 0.67, 12 1.00 / 0.69 / 0.69, 32 2.60 / 1.33 / 0.70; 64^2 x 12 0.74 / 0.70 / 0.75;
// 96^2, one problem 0.73 / 0.84 / 1.16, 16 1.81 / 1.27 / 1.17; 120^2 x 32 lossless
// 1.73 / 1.34 / 1.00.  (Counting rounds of resident clusters alone took 40^2 x 32
// in clusters of 8, behind the launched passes' 1.14.)
int choose(const LoopPlan& p, int batch) {
  // points of a CTA that take as long as the rest of a step
  const double flat = p.own_kernel ? 2600.0 : 6000.0;
  int k = -1;
  double best = 1e300;
  for (int q = 0; q < 3; ++q) {
    const int n = p.max_clusters[q];
    if (n <= 0) continue;
    const int rest = batch % n;
    const double full = n > p.alone[q] ? p.shared_cost : 1.0;
    const double rounds = batch / n * full + (rest == 0 ? 0.0 : rest > p.alone[q] ? full : 1.0);
    const double c = (1.0 + points_per_cta(p, q) / flat) * rounds;
    if (c < best) { best = c; k = q; }
  }
  return k;
}
}  // namespace

// (Where the launched passes are specialised on both axes they are the faster
// against smaller clusters of many points a CTA: 168^2 x 12 lossless, 24 steps,
// clusters of 8 with 3528 points 1.08 ms, launched 1.05; 168 x 48 x 24 lossless,
// clusters of 4 with 2016 0.99 / 0.89; 56^2 x 32, clusters of 4 with 784 0.76 / 1.30.)
int loop_waves(const LoopPlan& p, int batch) {
  const int k = choose(p, batch);
  if (k < 0 || (p.specialised && k > 0 && points_per_cta(p, k) > 1024.0)) return 1 << 30;
  return ceil_div(batch, p.max_clusters[k]);
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
