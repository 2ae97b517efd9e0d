// Diffusion-approximation optical solve (Section 2.1, eq. DA) in FP64.
//
// Cell-centred finite volumes on the interior grid (the optical grid is the
// acoustic interior): an interior face between cells a, b carries
// kappa_f (phi_a - phi_b) with the harmonic mean kappa_f (2D, the face
// length h cancels the 1/h of the gradient); the Robin condition
// phi + kappa/(2 gamma) dphi/dn = I/gamma, eliminated through the half-cell
// gradient, adds 2 gamma kappa h / (gamma h + kappa) to the diagonal and
// 2 kappa I h / (gamma h + kappa) to the right-hand side per boundary face;
// absorption adds mu h^2.  The matrix is symmetric positive definite and is
// solved by conjugate gradients preconditioned with one multigrid V-cycle (or the
// diagonal), with FP64 dot products (deterministic two-level reductions), batched
// over problems.
#include <algorithm>

#include "qpat_internal.h"

namespace qpat {

constexpr int kThreads = 256;

__device__ __forceinline__ double harmonic(double a, double b) { return 2.0 * a * b / (a + b); }

// Face, Robin and source coefficients of the finite-volume system for a
// grid of n0 x n1 x n2 cells (n2 = 1 in 2D): an interior face carries
// kappa_f h^(d-2), a boundary face adds 2 gamma kappa h^(d-1)/(gamma h + kappa)
// to the diagonal and 2 kappa I h^(d-1)/(gamma h + kappa) to the right-hand side.
__global__ void da_setup_kernel(int n0, int n1, int n2, int dim, double h, double gam, const double* kappa,
                                double* diag0, double* cxf, double* cyf, double* czf, double* bside) {
  const long long N = (long long)n0 * n1 * n2;
  const double hf = (dim == 3) ? h : 1.0;           // h^(d-2)
  const double hb = (dim == 3) ? h * h : h;         // h^(d-1)
  const long long sy = n0, sz = (long long)n0 * n1;
  for (long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x; g < N; g += (long long)gridDim.x * blockDim.x) {
    const int i = (int)(g % n0), j = (int)((g / n0) % n1), k = (int)(g / sz);
    const double kc = kappa[g];
    double d = 0.0;
    if (i > 0) d += harmonic(kc, kappa[g - 1]) * hf;
    if (i < n0 - 1) d += harmonic(kc, kappa[g + 1]) * hf;
    if (j > 0) d += harmonic(kc, kappa[g - sy]) * hf;
    if (j < n1 - 1) d += harmonic(kc, kappa[g + sy]) * hf;
    if (dim == 3) {
      if (k > 0) d += harmonic(kc, kappa[g - sz]) * hf;
      if (k < n2 - 1) d += harmonic(kc, kappa[g + sz]) * hf;
    }
    const double robin = 2.0 * gam * kc * hb / (gam * h + kc);
    const double src = 2.0 * kc * hb / (gam * h + kc);
    const bool on[6] = {i == 0, i == n0 - 1, j == 0, j == n1 - 1, dim == 3 && k == 0, dim == 3 && k == n2 - 1};
    for (int s = 0; s < 2 * dim; ++s) {
      if (on[s]) d += robin;
      bside[(long long)s * N + g] = on[s] ? src : 0.0;
    }
    diag0[g] = d;
    cxf[g] = (i < n0 - 1) ? harmonic(kc, kappa[g + 1]) * hf : 0.0;
    cyf[g] = (j < n1 - 1) ? harmonic(kc, kappa[g + sy]) * hf : 0.0;
    if (dim == 3) czf[g] = (k < n2 - 1) ? harmonic(kc, kappa[g + sz]) * hf : 0.0;
  }
}

cudaError_t da_setup(DAArgs& a, double* d_diag0, double* d_cxf, double* d_cyf, double* d_czf, double* d_bside,
                     const double* d_kappa, cudaStream_t s) {
  da_setup_kernel<<<256, kThreads, 0, s>>>(a.n0, a.n1, a.n2, a.dim, a.h, a.gamma, d_kappa, d_diag0, d_cxf, d_cyf,
                                           d_czf, d_bside);
  a.diag0 = d_diag0;
  a.cxf = d_cxf;
  a.cyf = d_cyf;
  a.czf = d_czf;
  a.bside = d_bside;
  return cudaGetLastError();
}

__global__ void rhs_sides_kernel(DAArgs a, unsigned mask, double* rhs) {
  const int b = blockIdx.y;
  const int sz = a.n0 * a.n1;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.N; g += gridDim.x * blockDim.x) {
    const int k = g / sz, rem = g - k * sz, j = rem / a.n0, i = rem - j * a.n0;
    const bool on[6] = {i == 0, i == a.n0 - 1, j == 0, j == a.n1 - 1, k == 0, k == a.n2 - 1};
    double v = 0.0;
#pragma unroll
    for (int s = 0; s < 6; ++s)                       // a side's coefficient is zero away from that side
      if (s < 2 * a.dim && on[s] && ((mask >> s) & 1u)) v += a.bside[(long long)s * a.N + g];
    rhs[(long long)b * a.N + g] = v;
  }
}

cudaError_t da_rhs_from_sides(const DAArgs& a, unsigned mask, int batch, double* rhs, cudaStream_t s) {
  rhs_sides_kernel<<<dim3((unsigned)std::min(kPCGBlocks, (a.N + kThreads - 1) / kThreads), batch), kThreads, 0, s>>>(a, mask,
                                                                                                                rhs);
  return cudaGetLastError();
}

__device__ __forceinline__ double apply_A(const DAArgs& a, const double* mu, const double* x, int g, double hd) {
  const int sy = a.n0, sz = a.n0 * a.n1;
  const int i = g % a.n0, j = (g / a.n0) % a.n1, k = g / sz;
  double y = (a.diag0[g] + mu[g] * hd) * x[g];
  if (i > 0) y -= a.cxf[g - 1] * x[g - 1];
  if (i < a.n0 - 1) y -= a.cxf[g] * x[g + 1];
  if (j > 0) y -= a.cyf[g - sy] * x[g - sy];
  if (j < a.n1 - 1) y -= a.cyf[g] * x[g + sy];
  if (a.dim == 3) {
    if (k > 0) y -= a.czf[g - sz] * x[g - sz];
    if (k < a.n2 - 1) y -= a.czf[g] * x[g + sz];
  }
  return y;
}

// Block-wide sum of up to 3 values, deterministic tree order; thread 0 writes.
__device__ __forceinline__ void block_sum3(double v0, double v1, double v2, double* out) {
  __shared__ double sh[3][kThreads];
  sh[0][threadIdx.x] = v0;
  sh[1][threadIdx.x] = v1;
  sh[2][threadIdx.x] = v2;
  __syncthreads();
  for (int st = kThreads / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) {
      sh[0][threadIdx.x] += sh[0][threadIdx.x + st];
      sh[1][threadIdx.x] += sh[1][threadIdx.x + st];
      sh[2][threadIdx.x] += sh[2][threadIdx.x + st];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    out[0] = sh[0][0];
    out[1] = sh[1][0];
    out[2] = sh[2][0];
  }
}

// scal layout per problem: [0] rz (even its), [1] rz (odd its), [2] pq, [3] rr, [4] bb, [5] done
__global__ void pcg_init_kernel(DAArgs a, const double* mu, const double* rhs, PCGWork w) {
  const int b = blockIdx.y;
  const long long o = (long long)b * a.N;
  const double h2 = a.hd;
  double rz = 0, rr = 0, bb = 0;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.N; g += gridDim.x * blockDim.x) {
    const double di = 1.0 / (a.diag0[g] + mu[o + g] * h2);
    const double r = rhs[o + g];
    w.dinv[o + g] = di;
    w.x[o + g] = 0.0;
    w.r[o + g] = r;
    w.z[o + g] = di * r;
    w.p[o + g] = di * r;
    rz += r * di * r;
    rr += r * r;
    bb += r * r;
  }
  block_sum3(rz, rr, bb, w.partial + ((long long)b * kPCGBlocks + blockIdx.x) * 4);
}

// Sum the partials of problem blockIdx.x into scal slots.
__global__ void pcg_reduce_kernel(PCGWork w, int s0, int s1, int s2) {
  const int b = blockIdx.x;
  const double* p = w.partial + (long long)b * kPCGBlocks * 4;
  double v0 = 0, v1 = 0, v2 = 0;
  for (int t = threadIdx.x; t < kPCGBlocks; t += blockDim.x) {
    v0 += p[4 * t];
    v1 += p[4 * t + 1];
    v2 += p[4 * t + 2];
  }
  __shared__ double res[3];
  block_sum3(v0, v1, v2, res);
  if (threadIdx.x == 0) {
    double* sc = w.scal + 8 * b;
    if (s0 >= 0) sc[s0] = res[0];
    if (s1 >= 0) sc[s1] = res[1];
    if (s2 >= 0) sc[s2] = res[2];
  }
}

__global__ void pcg_spmv_kernel(DAArgs a, const double* mu, PCGWork w) {
  const int b = blockIdx.y;
  const long long o = (long long)b * a.N;
  const double h2 = a.hd;
  double pq = 0;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.N; g += gridDim.x * blockDim.x) {
    const double q = apply_A(a, mu + o, w.p + o, g, h2);
    w.q[o + g] = q;
    pq += w.p[o + g] * q;
  }
  block_sum3(pq, 0.0, 0.0, w.partial + ((long long)b * kPCGBlocks + blockIdx.x) * 4);
}

__global__ void pcg_update_kernel(DAArgs a, PCGWork w, int parity) {
  const int b = blockIdx.y;
  const long long o = (long long)b * a.N;
  const double* sc = w.scal + 8 * b;
  const bool done = sc[5] != 0.0;
  const double rz = sc[parity], pq = sc[2];
  const double alpha = (done || pq == 0.0) ? 0.0 : rz / pq;
  double rz1 = 0, rr = 0;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.N; g += gridDim.x * blockDim.x) {
    const double x = w.x[o + g] + alpha * w.p[o + g];
    const double r = w.r[o + g] - alpha * w.q[o + g];
    const double z = w.dinv[o + g] * r;
    w.x[o + g] = x;
    w.r[o + g] = r;
    w.z[o + g] = z;
    rz1 += r * z;
    rr += r * r;
  }
  block_sum3(rz1, rr, 0.0, w.partial + ((long long)b * kPCGBlocks + blockIdx.x) * 4);
}

__global__ void pcg_pupdate_kernel(DAArgs a, PCGWork w, int parity) {
  const int b = blockIdx.y;
  const long long o = (long long)b * a.N;
  const double* sc = w.scal + 8 * b;
  const bool done = sc[5] != 0.0;
  const double rz_old = sc[parity], rz_new = sc[parity ^ 1];
  const double beta = (done || rz_old == 0.0) ? 0.0 : rz_new / rz_old;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.N; g += gridDim.x * blockDim.x)
    w.p[o + g] = w.z[o + g] + beta * w.p[o + g];
}

__global__ void pcg_mark_done_kernel(PCGWork w, int batch, double tol2) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  double* sc = w.scal + 8 * b;
  if (sc[3] <= tol2 * sc[4]) sc[5] = 1.0;
}

__global__ void copy_kernel(long long n, const double* in, double* out) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = in[t];
}

// ---- multigrid preconditioner ------------------------------------------------
// Cell-centred geometric multigrid on the same finite-volume discretisation:
// level l + 1 halves every axis of level l (while all are even and >= 4), its
// operator is rediscretised at spacing 2h from the children's mean kappa and
// mean mu, restriction sums the four (eight) children's residuals (R = P^T for
// the piecewise-constant prolongation P), smoothing is damped Jacobi with the
// same sweeps before and after the coarse correction, and the coarsest level
// gets a fixed number of Jacobi sweeps from zero.  Every step is linear and
// the V-cycle is symmetric, so it is a valid conjugate-gradient preconditioner.

__global__ void coarsen_mean_kernel(const double* f, double* c, int fn0, int fn1, int fn2, int dim, long long fstride,
                                    long long cstride) {
  const int b = blockIdx.y;
  const int cn0 = fn0 / 2, cn1 = fn1 / 2, cn2 = dim == 3 ? fn2 / 2 : 1;
  const long long Nc = (long long)cn0 * cn1 * cn2;
  const double inv = dim == 3 ? 0.125 : 0.25;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < Nc; t += (long long)gridDim.x * blockDim.x) {
    const int I = (int)(t % cn0), J = (int)((t / cn0) % cn1), K = (int)(t / ((long long)cn0 * cn1));
    double acc = 0.0;
    for (int dz = 0; dz < (dim == 3 ? 2 : 1); ++dz)
      for (int dy = 0; dy < 2; ++dy)
        for (int dx = 0; dx < 2; ++dx)
          acc += f[(long long)b * fstride + ((long long)(dim == 3 ? 2 * K + dz : 0) * fn1 + 2 * J + dy) * fn0 + 2 * I + dx];
    c[(long long)b * cstride + t] = acc * inv;
  }
}

cudaError_t mg_setup(MGHierarchy& h, const DAArgs& fine, const double* d_kappa, int max_batch, DevAlloc alloc,
                     void* owner, cudaStream_t s) {
  h.nlev = 1;
  h.lev[0].A = fine;
  h.lev[0].kappa = const_cast<double*>(d_kappa);
  const double* kap = d_kappa;
  while (h.nlev < kMaxLevels) {
    const DAArgs& f = h.lev[h.nlev - 1].A;
    const bool ok = f.n0 % 2 == 0 && f.n1 % 2 == 0 && f.n0 >= 4 && f.n1 >= 4 &&
                    (f.dim == 2 || (f.n2 % 2 == 0 && f.n2 >= 4));
    if (!ok) break;
    DAArgs c = f;
    c.n0 = f.n0 / 2;
    c.n1 = f.n1 / 2;
    c.n2 = f.dim == 3 ? f.n2 / 2 : 1;
    c.N = c.n0 * c.n1 * c.n2;
    c.h = 2.0 * f.h;
    c.hd = f.dim == 3 ? c.h * c.h * c.h : c.h * c.h;
    double *ck, *d0, *cx, *cy, *cz, *bs;
    cudaError_t e;
    if ((e = alloc(owner, (void**)&ck, c.N * sizeof(double))) != cudaSuccess) return e;
    coarsen_mean_kernel<<<dim3(128, 1), kThreads, 0, s>>>(kap, ck, f.n0, f.n1, f.n2, f.dim, 0, 0);
    for (double** p : {&d0, &cx, &cy, &cz})
      if ((e = alloc(owner, (void**)p, c.N * sizeof(double))) != cudaSuccess) return e;
    if ((e = alloc(owner, (void**)&bs, (size_t)2 * c.dim * c.N * sizeof(double))) != cudaSuccess) return e;
    if ((e = da_setup(c, d0, cx, cy, cz, bs, ck, s)) != cudaSuccess) return e;
    h.lev[h.nlev].A = c;
    h.lev[h.nlev].kappa = ck;
    kap = ck;
    ++h.nlev;
  }
  for (int l = 0; l < h.nlev; ++l) {
    // one allocation a level (each takes some tenths of a millisecond); level 0
    // uses the PCG work vectors but for x2
    MGLevel& L = h.lev[l];
    const size_t n = ((size_t)max_batch * L.A.N + 1) & ~(size_t)1;   // 16-byte multiples
    double* v = nullptr;
    const cudaError_t e = alloc(owner, (void**)&v, (l > 0 ? 6 : 1) * n * sizeof(double));
    if (e != cudaSuccess) return e;
    L.x2 = v;
    if (l > 0) {
      L.mu = v + n;
      L.x = v + 2 * n;
      L.b = v + 3 * n;
      L.d = v + 4 * n;
      L.w = v + 5 * n;
    }
  }
  return cudaGetLastError();
}

cudaError_t mg_rekappa(MGHierarchy& h, cudaStream_t s) {
  for (int l = 1; l < h.nlev; ++l) {
    const DAArgs& f = h.lev[l - 1].A;
    DAArgs& c = h.lev[l].A;
    coarsen_mean_kernel<<<dim3(128, 1), kThreads, 0, s>>>(h.lev[l - 1].kappa, h.lev[l].kappa, f.n0, f.n1, f.n2, f.dim,
                                                          0, 0);
    cudaError_t e = da_setup(c, const_cast<double*>(c.diag0), const_cast<double*>(c.cxf),
                             const_cast<double*>(c.cyf), const_cast<double*>(c.czf), const_cast<double*>(c.bside),
                             h.lev[l].kappa, s);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

// ---- V-cycle and multigrid-preconditioned iteration ----------------------------
// GB300 has two FP64 fused multiply-adds per clock and SM, so on large grids
// these kernels are bound by FP64 arithmetic as much as by memory, and on
// small ones by the number of launches.  Hence: the smoother multiplies by a
// stored omega / d instead of dividing (a division is about ten FP64
// instructions; a sweep is 2 dim + 2); the first sweep from zero is part of
// the kernel that makes the right-hand side, the prolongation part of the
// coarse level's last sweep, and every inner product is finished by the last
// block of the kernel that forms it; a thread takes two adjacent cells with
// 16-byte loads; all levels of at most kSmallCells cells run in one CTA per
// problem, in shared memory; and a converged problem's blocks return at once.
// Measured on GB300: 512^2, 8 problems 12.2 -> 4.9 ms; 128^2, one problem 2.6 -> 1.3 ms; 90^2
// (stops at 45^2) 14.7 -> 3.2 ms; the forward map on 256^3 with 24 time steps 130 -> 81 ms.

// One level of one solve, as the kernels see it.
struct LevDev {
  int n0, n1, n2, N;
  const double *cx, *cy, *cz, *d, *w;
  double *x, *x2, *b;
};

static LevDev mg_dev(const MGLevel& L, const PCGWork&) {
  return LevDev{L.A.n0, L.A.n1, L.A.n2, L.A.N, L.A.cxf, L.A.cyf, L.A.czf, L.d, L.w, L.x, L.x2, L.b};
}

// Launch shape of a level: TX x TY threads, a thread taking VEC adjacent cells
// of a grid line (VEC = 2 where lines are even), blocks striding over lines.
// It depends on the level only, so a problem's sums are the same in any batch.
struct MGGrid {
  dim3 grid, block;
  int vec;
};
static MGGrid mg_grid(const DAArgs& a, int batch) {
  MGGrid g;
  g.vec = a.n0 % 2 == 0 ? 2 : 1;
  int tx = 8;
  while (tx < 64 && tx < a.n0 / g.vec) tx *= 2;
  const int ty = kThreads / tx, lines = a.n1 * a.n2;
  g.block = dim3(tx, ty);
  g.grid = dim3((unsigned)std::min(kPCGBlocks, (lines + ty - 1) / ty), batch);
  return g;
}
static dim3 mg_blocks(int N, int batch) {
  return dim3((unsigned)std::min(kPCGBlocks, (N + kThreads - 1) / kThreads), batch);
}
#define MG_DISPATCH(A_, kernel, g_, s_, ...)                                                \
  do {                                                                                      \
    if ((A_).dim == 3) {                                                                    \
      if ((g_).vec == 2) kernel<3, 2><<<(g_).grid, (g_).block, 0, s_>>>(__VA_ARGS__);       \
      else kernel<3, 1><<<(g_).grid, (g_).block, 0, s_>>>(__VA_ARGS__);                     \
    } else {                                                                                \
      if ((g_).vec == 2) kernel<2, 2><<<(g_).grid, (g_).block, 0, s_>>>(__VA_ARGS__);       \
      else kernel<2, 1><<<(g_).grid, (g_).block, 0, s_>>>(__VA_ARGS__);                     \
    }                                                                                       \
  } while (0)

template <int VEC>
struct Cells {
  double v[VEC];
};
template <int VEC>
__device__ __forceinline__ Cells<VEC> ld(const double* p) {
  Cells<VEC> c;
  if constexpr (VEC == 2) {
    const double2 t = *reinterpret_cast<const double2*>(p);
    c.v[0] = t.x;
    c.v[1] = t.y;
  } else {
    c.v[0] = *p;
  }
  return c;
}
template <int VEC>
__device__ __forceinline__ void st(double* p, const Cells<VEC>& c) {
  if constexpr (VEC == 2) *reinterpret_cast<double2*>(p) = make_double2(c.v[0], c.v[1]);
  else *p = c.v[0];
}

// body(g, i, j, k) for the VEC-cell groups of a level of blockIdx.y's problem.
template <int DIM, int VEC, class F>
__device__ __forceinline__ void for_groups(int n0, int n1, int n2, F&& body) {
  const int lines = n1 * n2;
  for (int line = blockIdx.x * blockDim.y + threadIdx.y; line < lines; line += gridDim.x * blockDim.y) {
    const int k = DIM == 3 ? line / n1 : 0, j = DIM == 3 ? line - k * n1 : line;
    for (int i = threadIdx.x * VEC; i < n0; i += blockDim.x * VEC) body(line * n0 + i, i, j, k);
  }
}

// c - A x at the VEC cells from g = (i, j, k); X receives x there.
template <int DIM, int VEC>
__device__ __forceinline__ Cells<VEC> residual(const LevDev& L, const double* d, const double* x, Cells<VEC> c, int g,
                                               int i, int j, int k, Cells<VEC>& X) {
  const int sy = L.n0, sz = L.n0 * L.n1;
  X = ld<VEC>(x + g);
  const Cells<VEC> D = ld<VEC>(d + g), cr = ld<VEC>(L.cx + g);
  const double cl = i > 0 ? L.cx[g - 1] : 0.0, xl = i > 0 ? x[g - 1] : 0.0;
  const double xr = i + VEC < L.n0 ? x[g + VEC] : 0.0;
#pragma unroll
  for (int v = 0; v < VEC; ++v) {
    c.v[v] -= D.v[v] * X.v[v];
    c.v[v] += (v ? cr.v[0] : cl) * (v ? X.v[0] : xl);
    c.v[v] += cr.v[v] * (v + 1 < VEC ? X.v[VEC - 1] : xr);       // (zero coefficient at the last cell of a line)
  }
  if (j > 0) {
    const Cells<VEC> f = ld<VEC>(L.cy + g - sy), y = ld<VEC>(x + g - sy);
#pragma unroll
    for (int v = 0; v < VEC; ++v) c.v[v] += f.v[v] * y.v[v];
  }
  if (j < L.n1 - 1) {
    const Cells<VEC> f = ld<VEC>(L.cy + g), y = ld<VEC>(x + g + sy);
#pragma unroll
    for (int v = 0; v < VEC; ++v) c.v[v] += f.v[v] * y.v[v];
  }
  if (DIM == 3) {
    if (k > 0) {
      const Cells<VEC> f = ld<VEC>(L.cz + g - sz), y = ld<VEC>(x + g - sz);
#pragma unroll
      for (int v = 0; v < VEC; ++v) c.v[v] += f.v[v] * y.v[v];
    }
    if (k < L.n2 - 1) {
      const Cells<VEC> f = ld<VEC>(L.cz + g), y = ld<VEC>(x + g + sz);
#pragma unroll
      for (int v = 0; v < VEC; ++v) c.v[v] += f.v[v] * y.v[v];
    }
  }
  return c;
}

// Sum v over the launch's blocks of problem blockIdx.y, in a fixed order: true
// (with the total in v) in thread 0 of the block that finishes last.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((tid & 31) == 0) sh[tid >> 5] = v;
  __syncthreads();
  double t = 0.0;
  if (tid == 0)
    for (int q = 0; q < kThreads / 32; ++q) t += sh[q];
  return t;
}
__device__ __forceinline__ bool last_block_sum(double& v, const PCGWork& w) {
  __shared__ double sh[kThreads / 32], sh2[kThreads / 32];
  __shared__ bool last;
  const int tid = threadIdx.y * blockDim.x + threadIdx.x, b = blockIdx.y;
  double* part = w.partial + (long long)b * kPCGBlocks * 4;
  const double t = block_sum(v, sh);
  if (tid == 0) {
    part[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(&w.count[b], 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double u = 0.0;
  for (int q = tid; q < (int)gridDim.x; q += kThreads) u += __ldcg(part + q);
  v = block_sum(u, sh2);
  if (tid == 0) w.count[b] = 0;
  return tid == 0;
}
__device__ __forceinline__ bool pcg_done(const PCGWork& w) { return w.scal[8 * blockIdx.y + 5] != 0.0; }

// d = diag0 + mu h^dim and omega / d of a level.
__global__ void mg_diag_kernel(DAArgs a, const double* mu, double omega, double* d, double* w) {
  const long long o = (long long)blockIdx.y * a.N;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.N; g += gridDim.x * blockDim.x) {
    const double v = a.diag0[g] + mu[o + g] * a.hd;
    d[o + g] = v;
    w[o + g] = omega / v;
  }
}
// The same on the next level, whose absorption is the mean of the children's.
__global__ void mg_coarsen_kernel(DAArgs f, DAArgs c, const double* muf, double omega, double* muc, double* d,
                                  double* w) {
  const long long of = (long long)blockIdx.y * f.N, oc = (long long)blockIdx.y * c.N;
  const double inv = f.dim == 3 ? 0.125 : 0.25;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < c.N; t += gridDim.x * blockDim.x) {
    const int I = t % c.n0, J = (t / c.n0) % c.n1, K = t / (c.n0 * c.n1);
    double acc = 0.0;
    for (int dz = 0; dz < (f.dim == 3 ? 2 : 1); ++dz)
      for (int dy = 0; dy < 2; ++dy)
        for (int dx = 0; dx < 2; ++dx)
          acc += muf[of + ((long long)(f.dim == 3 ? 2 * K + dz : 0) * f.n1 + 2 * J + dy) * f.n0 + 2 * I + dx];
    const double m = acc * inv, v = c.diag0[t] + m * c.hd;
    muc[oc + t] = m;
    d[oc + t] = v;
    w[oc + t] = omega / v;
  }
}

// out = x + w (b - A x).  DOT: b . out into scal[slot] (level 0: r.z).
// PROLONG: the result is not stored but added to its children in xf.
enum SweepMode { kSweep, kSweepDot, kSweepProlong };
template <int DIM, int VEC, int MODE>
__device__ __forceinline__ void sweep_body(const LevDev& L, const double* xin, double* out, const PCGWork& w, int slot,
                                           double* xf) {
  if (pcg_done(w)) return;
  const long long o = (long long)blockIdx.y * L.N;
  const double *x = xin + o, *d = L.d + o;
  double dot = 0.0;
  for_groups<DIM, VEC>(L.n0, L.n1, L.n2, [&](int g, int i, int j, int k) {
    const Cells<VEC> b = ld<VEC>(L.b + o + g), wd = ld<VEC>(L.w + o + g);
    Cells<VEC> X, r = residual<DIM, VEC>(L, d, x, b, g, i, j, k, X);
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      r.v[v] = X.v[v] + wd.v[v] * r.v[v];
      if (MODE == kSweepDot) dot += b.v[v] * r.v[v];
    }
    if (MODE != kSweepProlong) {
      st<VEC>(out + o + g, r);
    } else {
      const int f0 = 2 * L.n0, f1 = 2 * L.n1;
      double* f = xf + (long long)blockIdx.y * L.N * (DIM == 3 ? 8 : 4);
#pragma unroll
      for (int v = 0; v < VEC; ++v)
        for (int dz = 0; dz < (DIM == 3 ? 2 : 1); ++dz)
          for (int dy = 0; dy < 2; ++dy) {
            double2* q = reinterpret_cast<double2*>(f + ((long long)(DIM == 3 ? 2 * k + dz : 0) * f1 + 2 * j + dy) * f0 +
                                                    2 * (i + v));
            double2 t = *q;
            t.x += r.v[v];
            t.y += r.v[v];
            *q = t;
          }
    }
  });
  if (MODE == kSweepDot) {
    if (last_block_sum(dot, w)) w.scal[8 * blockIdx.y + slot] = dot;
  }
}
template <int DIM, int VEC>
__global__ void __launch_bounds__(kThreads) mg_sweep(LevDev L, const double* xin, double* out, PCGWork w) {
  sweep_body<DIM, VEC, kSweep>(L, xin, out, w, 0, nullptr);
}
template <int DIM, int VEC>
__global__ void __launch_bounds__(kThreads) mg_sweep_dot(LevDev L, const double* xin, double* out, PCGWork w, int slot) {
  sweep_body<DIM, VEC, kSweepDot>(L, xin, out, w, slot, nullptr);
}
template <int DIM, int VEC>
__global__ void __launch_bounds__(kThreads) mg_sweep_prolong(LevDev L, const double* xin, double* xf, PCGWork w) {
  sweep_body<DIM, VEC, kSweepProlong>(L, xin, nullptr, w, 0, xf);
}

// b_c = sum over the children of (b - A x), and the first sweep from zero
// there, x2_c = w_c b_c.  A thread takes one coarse cell (fine lines are even).
template <int DIM>
__global__ void __launch_bounds__(kThreads) mg_restrict(LevDev F, LevDev C, PCGWork w) {
  if (pcg_done(w)) return;
  const long long of = (long long)blockIdx.y * F.N, oc = (long long)blockIdx.y * C.N;
  for_groups<DIM, 1>(C.n0, C.n1, C.n2, [&](int t, int I, int J, int K) {
    double acc = 0.0;
#pragma unroll
    for (int dz = 0; dz < (DIM == 3 ? 2 : 1); ++dz)
#pragma unroll
      for (int dy = 0; dy < 2; ++dy) {
        const int k = DIM == 3 ? 2 * K + dz : 0, j = 2 * J + dy, i = 2 * I;
        const int g = (k * F.n1 + j) * F.n0 + i;
        Cells<2> X;
        const Cells<2> r = residual<DIM, 2>(F, F.d + of, F.x + of, ld<2>(F.b + of + g), g, i, j, k, X);
        acc += r.v[0] + r.v[1];
      }
    C.b[oc + t] = acc;
    C.x2[oc + t] = C.w[oc + t] * acc;
  });
}

// The levels of at most kSmallCells cells, of one problem in one CTA: the
// whole V-cycle from the right-hand side b of the first of them, in shared
// memory, the result added to its children in xf.
constexpr int kSmallCells = 512;
constexpr int kMaxSmall = 6;
struct SmallLevels {
  int n, dim, sweeps;                  // levels; sweeps of the coarsest
  LevDev lev[kMaxSmall];
  double* xf;
};
static size_t small_smem(const SmallLevels& S) {
  size_t t = 0;
  for (int l = 0; l < S.n; ++l) t += (size_t)S.lev[l].N * 8;
  return t * sizeof(double);
}
// A level in shared memory: x and a second buffer t, b, d, w, and the face
// coefficients cx, cy, cz.
struct SmallLev {
  double *x, *t, *b, *d, *w, *cx, *cy, *cz;
};
// Cell g with the offsets of its neighbours and their coefficients' (an absent
// neighbour reads the cell itself with coefficient 0), worked out once per cell
// and level: the sweeps have no index arithmetic left.
struct SmallCell {
  double cl, cr, cd, cu, cb, cf, d, w, b;
  int il, ir, id, iu, ib, jf;
};
template <int DIM>
__device__ __forceinline__ SmallCell small_cell(const LevDev& L, const SmallLev& s, int g) {
  const int sy = L.n0, sz = L.n0 * L.n1;
  const int k = DIM == 3 ? g / sz : 0, rem = g - k * sz, j = rem / L.n0, i = rem - j * L.n0;
  SmallCell c;
  c.il = i > 0 ? g - 1 : g;
  c.cl = i > 0 ? s.cx[g - 1] : 0.0;
  c.ir = i < L.n0 - 1 ? g + 1 : g;
  c.cr = i < L.n0 - 1 ? s.cx[g] : 0.0;
  c.id = j > 0 ? g - sy : g;
  c.cd = j > 0 ? s.cy[g - sy] : 0.0;
  c.iu = j < L.n1 - 1 ? g + sy : g;
  c.cu = j < L.n1 - 1 ? s.cy[g] : 0.0;
  if (DIM == 3) {
    c.ib = k > 0 ? g - sz : g;
    c.cb = k > 0 ? s.cz[g - sz] : 0.0;
    c.jf = k < L.n2 - 1 ? g + sz : g;
    c.cf = k < L.n2 - 1 ? s.cz[g] : 0.0;
  }
  c.d = s.d[g];
  c.w = s.w[g];
  c.b = s.b[g];
  return c;
}
// b - A x at cell g, as two chains of fused multiply-adds.
template <int DIM>
__device__ __forceinline__ double small_res(const SmallCell& c, const double* x, int g) {
  double r = c.b - c.d * x[g];
  double u = c.cd * x[c.id] + c.cu * x[c.iu];
  r += c.cl * x[c.il];
  r += c.cr * x[c.ir];
  if (DIM == 3) {
    u += c.cb * x[c.ib];
    u += c.cf * x[c.jf];
  }
  return r + u;
}
// The cells of this thread on one level (kSmallCells / kThreads of them).
constexpr int kSmallPer = (kSmallCells + kThreads - 1) / kThreads;
template <int DIM>
struct SmallCells {
  SmallCell c[kSmallPer];
  int N;
  __device__ __forceinline__ SmallCells(const LevDev& L, const SmallLev& s) : N(L.N) {
    each([&](int q, int g) { c[q] = small_cell<DIM>(L, s, g); });
  }
  template <class F>
  __device__ __forceinline__ void each(F&& f) {
#pragma unroll
    for (int q = 0; q < kSmallPer; ++q)
      if ((int)threadIdx.x + q * kThreads < N) f(q, (int)threadIdx.x + q * kThreads);
  }
  __device__ __forceinline__ void sweep(const double* in, double* out) {
    each([&](int q, int g) { out[g] = in[g] + c[q].w * small_res<DIM>(c[q], in, g); });
    __syncthreads();
  }
};
// The V-cycle over the levels of S (b of the first is set), x of the first
// receiving the result.
template <int DIM>
__device__ __forceinline__ void small_cycle(const SmallLevels& S, const SmallLev* sl) {
  const int tid = threadIdx.x;
  for (int l = 0; l + 1 < S.n; ++l) {
    const LevDev &L = S.lev[l], &C = S.lev[l + 1];
    const SmallLev s = sl[l];
    SmallCells<DIM> c(L, s);
    c.each([&](int q, int g) { s.t[g] = c.c[q].w * c.c[q].b; });
    __syncthreads();
    c.sweep(s.t, s.x);
    // the residual of every cell, then its sum over the children of each coarse cell
    c.each([&](int q, int g) { s.t[g] = small_res<DIM>(c.c[q], s.x, g); });
    __syncthreads();
    for (int t = tid; t < C.N; t += kThreads) {
      const int K = DIM == 3 ? t / (C.n0 * C.n1) : 0, rem = t - K * C.n0 * C.n1, J = rem / C.n0, I = rem - J * C.n0;
      double acc = 0.0;
      for (int dz = 0; dz < (DIM == 3 ? 2 : 1); ++dz)
        for (int dy = 0; dy < 2; ++dy) {
          const double* f = s.t + ((DIM == 3 ? 2 * K + dz : 0) * L.n1 + 2 * J + dy) * L.n0 + 2 * I;
          acc += f[0] + f[1];
        }
      sl[l + 1].b[t] = acc;
    }
    __syncthreads();
  }
  {
    // the coarsest level: an odd number of sweeps from zero, the result in x; a
    // level of at most 32 cells stays in one warp
    const LevDev& L = S.lev[S.n - 1];
    const SmallLev s = sl[S.n - 1];
    SmallCells<DIM> c(L, s);
    c.each([&](int q, int g) { s.x[g] = c.c[q].w * c.c[q].b; });
    __syncthreads();
    if (L.N > 32) {
      for (int q = 1; q < S.sweeps; q += 2) {
        c.sweep(s.x, s.t);
        c.sweep(s.t, s.x);
      }
    } else {
      if (tid < 32) {
        for (int q = 1; q < S.sweeps; q += 2) {
          if (tid < L.N) s.t[tid] = s.x[tid] + c.c[0].w * small_res<DIM>(c.c[0], s.x, tid);
          __syncwarp();
          if (tid < L.N) s.x[tid] = s.t[tid] + c.c[0].w * small_res<DIM>(c.c[0], s.t, tid);
          __syncwarp();
        }
      }
      __syncthreads();
    }
  }
  for (int l = S.n - 2; l >= 0; --l) {
    const LevDev &L = S.lev[l], &C = S.lev[l + 1];
    const SmallLev s = sl[l];
    const double* xc = sl[l + 1].x;
    SmallCells<DIM> c(L, s);
    c.each([&](int, int g) {
      const int k = DIM == 3 ? g / (L.n0 * L.n1) : 0, rem = g - k * L.n0 * L.n1, j = rem / L.n0, i = rem - j * L.n0;
      s.x[g] += xc[((DIM == 3 ? k >> 1 : 0) * C.n1 + (j >> 1)) * C.n0 + (i >> 1)];
    });
    __syncthreads();
    c.sweep(s.x, s.t);
    c.sweep(s.t, s.x);
  }
}
template <int DIM>
__global__ void __launch_bounds__(kThreads) mg_small(const __grid_constant__ SmallLevels S, PCGWork w) {
  extern __shared__ __align__(16) double sm[];
  if (w.scal[8 * blockIdx.x + 5] != 0.0) return;
  const int tid = threadIdx.x;
  __shared__ SmallLev sl[kMaxSmall];
  if (tid == 0) {
    double* p = sm;
    for (int l = 0; l < S.n; ++l) {
      const int N = S.lev[l].N;
      sl[l] = SmallLev{p, p + N, p + 2 * N, p + 3 * N, p + 4 * N, p + 5 * N, p + 6 * N, p + 7 * N};
      p += 8 * N;
    }
  }
  __syncthreads();
  for (int l = 0; l < S.n; ++l) {
    const LevDev& L = S.lev[l];
    const SmallLev s = sl[l];
    const long long o = (long long)blockIdx.x * L.N;
    for (int g = tid; g < L.N; g += kThreads) {
      if (l == 0) s.b[g] = L.b[o + g];
      s.d[g] = L.d[o + g];
      s.w[g] = L.w[o + g];
      s.cx[g] = L.cx[g];
      s.cy[g] = L.cy[g];
      if (DIM == 3) s.cz[g] = L.cz[g];
    }
  }
  __syncthreads();
  small_cycle<DIM>(S, sl);
  const LevDev& L = S.lev[0];
  const int f0 = 2 * L.n0, f1 = 2 * L.n1, Nf = L.N * (DIM == 3 ? 8 : 4);
  double* f = S.xf + (long long)blockIdx.x * Nf;
  for (int g = tid; g < Nf; g += kThreads) {
    const int k = g / (f0 * f1), rem = g - k * f0 * f1, j = rem / f0, i = rem - j * f0;
    f[g] += sl[0].x[((DIM == 3 ? k >> 1 : 0) * L.n1 + (j >> 1)) * L.n0 + (i >> 1)];
  }
}

// All sweeps of a coarsest level above kSmallCells (a grid whose extents turn
// odd early): eight CTAs of one cluster per problem, a cluster barrier between
// sweeps (a launch per sweep took 41 launches), the result added to its
// children in xf.
constexpr int kClusterCells = 8192, kCoarseCluster = 8, kCoarseThreads = 512;
__device__ __forceinline__ void coarse_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__global__ void __cluster_dims__(kCoarseCluster, 1, 1) __launch_bounds__(kCoarseThreads)
mg_coarse_cluster(LevDev L, double* xf, PCGWork w, int dim, int sweeps) {
  const int b = blockIdx.x / kCoarseCluster;
  if (w.scal[8 * b + 5] != 0.0) return;                          // (the whole cluster: one problem)
  const long long o = (long long)b * L.N;
  const int per = (L.N + kCoarseCluster - 1) / kCoarseCluster;
  const int g0 = (blockIdx.x % kCoarseCluster) * per, g1 = min(L.N, g0 + per);
  const int sy = L.n0, sz = L.n0 * L.n1;
  double *cur = L.x2 + o, *nxt = L.x + o;                        // x2 = w b is there already
  for (int q = 1; q < sweeps; ++q) {
    for (int g = g0 + threadIdx.x; g < g1; g += kCoarseThreads) {
      const int k = g / sz, rem = g - k * sz, j = rem / L.n0, i = rem - j * L.n0;
      const double x = __ldcg(cur + g);
      double r = L.b[o + g] - L.d[o + g] * x;
      if (i > 0) r += L.cx[g - 1] * __ldcg(cur + g - 1);
      if (i < L.n0 - 1) r += L.cx[g] * __ldcg(cur + g + 1);
      if (j > 0) r += L.cy[g - sy] * __ldcg(cur + g - sy);
      if (j < L.n1 - 1) r += L.cy[g] * __ldcg(cur + g + sy);
      if (dim == 3) {
        if (k > 0) r += L.cz[g - sz] * __ldcg(cur + g - sz);
        if (k < L.n2 - 1) r += L.cz[g] * __ldcg(cur + g + sz);
      }
      nxt[g] = x + L.w[o + g] * r;
    }
    coarse_sync();
    double* t = cur;
    cur = nxt;
    nxt = t;
  }
  const int f0 = 2 * L.n0, f1 = 2 * L.n1, nch = dim == 3 ? 4 : 2;
  double* f = xf + (long long)b * L.N * (dim == 3 ? 8 : 4);
  for (int g = g0 + threadIdx.x; g < g1; g += kCoarseThreads) {
    const int k = g / sz, rem = g - k * sz, j = rem / L.n0, i = rem - j * L.n0;
    const double v = __ldcg(cur + g);
    for (int q = 0; q < nch; ++q) {
      double* p = f + ((long long)(dim == 3 ? 2 * k + (q >> 1) : 0) * f1 + 2 * j + (q & 1)) * f0 + 2 * i;
      p[0] += v;
      p[1] += v;
    }
  }
}

// First level (at least 1) from which all levels fit mg_small; nlev if none.
static int small_from(const MGHierarchy& h) {
  int l = h.nlev;
  size_t cells = 0;
  while (l > 1 && h.lev[l - 1].A.N <= kSmallCells && h.nlev - l < kMaxSmall) cells += h.lev[--l].A.N;
  return l;
}

// z = V-cycle(r): r.z goes to scal[slot].  Level 0's x2 = w r is there already.
static void mg_vcycle(MGHierarchy& h, PCGWork& w, int batch, int slot, cudaStream_t s) {
  const int ls = small_from(h), dim = h.lev[0].A.dim;
  const int bottom = ls < h.nlev ? ls : h.nlev - 1;              // first level not smoothed by launches of its own
  for (int l = 0; l < bottom; ++l) {
    const LevDev L = mg_dev(h.lev[l], w), C = mg_dev(h.lev[l + 1], w);
    const MGGrid g = mg_grid(h.lev[l].A, batch);
    MG_DISPATCH(h.lev[l].A, mg_sweep, g, s, L, L.x2, L.x, w);
    MGGrid gc = mg_grid(h.lev[l + 1].A, batch);
    if (dim == 3) mg_restrict<3><<<gc.grid, gc.block, 0, s>>>(L, C, w);
    else mg_restrict<2><<<gc.grid, gc.block, 0, s>>>(L, C, w);
  }
  const MGLevel& B = h.lev[bottom];
  double* xf = h.lev[bottom - 1].x;
  if (ls < h.nlev) {
    SmallLevels S{};
    S.n = h.nlev - ls;
    S.dim = dim;
    S.sweeps = h.coarse_sweeps;
    for (int l = ls; l < h.nlev; ++l) S.lev[l - ls] = mg_dev(h.lev[l], w);
    S.xf = xf;
    if (dim == 3) mg_small<3><<<batch, kThreads, small_smem(S), s>>>(S, w);
    else mg_small<2><<<batch, kThreads, small_smem(S), s>>>(S, w);
  } else if (B.A.N <= kClusterCells) {
    mg_coarse_cluster<<<kCoarseCluster * batch, kCoarseThreads, 0, s>>>(mg_dev(B, w), xf, w, dim, h.coarse_sweeps);
  } else {
    const LevDev L = mg_dev(B, w);
    const MGGrid g = mg_grid(B.A, batch);
    double *cur = L.x2, *nxt = L.x;
    for (int it = 1; it + 1 < h.coarse_sweeps; ++it) {
      MG_DISPATCH(B.A, mg_sweep, g, s, L, cur, nxt, w);
      std::swap(cur, nxt);
    }
    MG_DISPATCH(B.A, mg_sweep_prolong, g, s, L, cur, xf, w);
  }
  for (int l = bottom - 1; l >= 0; --l) {
    const LevDev L = mg_dev(h.lev[l], w);
    const MGGrid g = mg_grid(h.lev[l].A, batch);
    MG_DISPATCH(h.lev[l].A, mg_sweep, g, s, L, L.x, L.x2, w);
    if (l == 0) MG_DISPATCH(h.lev[l].A, mg_sweep_dot, g, s, L, L.x2, L.x, w, slot);
    else MG_DISPATCH(h.lev[l].A, mg_sweep_prolong, g, s, L, L.x2, h.lev[l - 1].x, w);
  }
}

// The vectors of one problem as [0, N) in pairs of cells: body(t) for t = 0, 2, ...
template <class F>
__device__ __forceinline__ void for_pairs(int N, F&& body) {
  const int tid = threadIdx.y * blockDim.x + threadIdx.x;
  for (int t = 2 * (blockIdx.x * kThreads + tid); t < N; t += 2 * (int)gridDim.x * kThreads) body(t);
}

// x = 0, r = rhs, the first sweep of the V-cycle, bb = rr = rhs.rhs
__global__ void __launch_bounds__(kThreads) pcg_init_mg(int N, const double* rhs, PCGWork w) {
  const long long o = (long long)blockIdx.y * N;
  double *x = w.x + o, *r = w.r + o, *x2 = w.mg_x2 + o;
  const double *q = rhs + o, *wd = w.dinv + o;
  double rr = 0.0;
  for_pairs(N, [&](int t) {                                      // (N is even: mg needs even extents)
    const Cells<2> v = ld<2>(q + t), m = ld<2>(wd + t);
    st<2>(x + t, Cells<2>{{0.0, 0.0}});
    st<2>(r + t, v);
    st<2>(x2 + t, Cells<2>{{m.v[0] * v.v[0], m.v[1] * v.v[1]}});
    rr += v.v[0] * v.v[0] + v.v[1] * v.v[1];
  });
  if (last_block_sum(rr, w)) {
    w.scal[8 * blockIdx.y + 3] = rr;
    w.scal[8 * blockIdx.y + 4] = rr;
  }
}

// q = A p, p.q
template <int DIM, int VEC>
__global__ void __launch_bounds__(kThreads) pcg_spmv_mg(LevDev L, PCGWork w) {
  if (pcg_done(w)) return;
  const long long o = (long long)blockIdx.y * L.N;
  double pq = 0.0;
  for_groups<DIM, VEC>(L.n0, L.n1, L.n2, [&](int g, int i, int j, int k) {
    Cells<VEC> X, r;
#pragma unroll
    for (int v = 0; v < VEC; ++v) r.v[v] = 0.0;
    r = residual<DIM, VEC>(L, L.d + o, w.p + o, r, g, i, j, k, X);
#pragma unroll
    for (int v = 0; v < VEC; ++v) {
      r.v[v] = -r.v[v];
      pq += X.v[v] * r.v[v];
    }
    st<VEC>(w.q + o + g, r);
  });
  if (last_block_sum(pq, w)) w.scal[8 * blockIdx.y + 2] = pq;
}

// x += alpha p, r -= alpha q, the first sweep of the V-cycle on r, r.r, and the
// convergence flag
__global__ void __launch_bounds__(kThreads) pcg_update_mg(int N, PCGWork w, int parity, double tol2) {
  double* sc = w.scal + 8 * blockIdx.y;
  if (sc[5] != 0.0) return;
  const long long o = (long long)blockIdx.y * N;
  double *x = w.x + o, *r = w.r + o, *x2 = w.mg_x2 + o;
  const double *p = w.p + o, *q = w.q + o, *wd = w.dinv + o;
  const double rz = sc[parity], pq = sc[2];
  const double alpha = pq == 0.0 ? 0.0 : rz / pq;
  double rr = 0.0;
  for_pairs(N, [&](int t) {
    Cells<2> X = ld<2>(x + t), R = ld<2>(r + t), M = ld<2>(wd + t);
    const Cells<2> P = ld<2>(p + t), Q = ld<2>(q + t);
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      X.v[v] += alpha * P.v[v];
      R.v[v] -= alpha * Q.v[v];
      M.v[v] *= R.v[v];
      rr += R.v[v] * R.v[v];
    }
    st<2>(x + t, X);
    st<2>(r + t, R);
    st<2>(x2 + t, M);
  });
  if (last_block_sum(rr, w)) {
    sc[3] = rr;
    if (rr <= tol2 * sc[4]) sc[5] = 1.0;
  }
}

// p = z + beta p (first: p = z)
__global__ void __launch_bounds__(kThreads) pcg_pupdate_mg(int N, PCGWork w, int parity, int first) {
  const double* sc = w.scal + 8 * blockIdx.y;
  if (sc[5] != 0.0) return;
  const long long o = (long long)blockIdx.y * N;
  double* p = w.p + o;
  const double* z = w.z + o;
  const double rz_old = sc[parity], rz_new = sc[parity ^ 1];
  const double beta = (first || rz_old == 0.0) ? 0.0 : rz_new / rz_old;
  for_pairs(N, [&](int t) {
    Cells<2> Z = ld<2>(z + t);
    if (!first) {
      const Cells<2> P = ld<2>(p + t);
#pragma unroll
      for (int v = 0; v < 2; ++v) Z.v[v] += beta * P.v[v];
    }
    st<2>(p + t, Z);
  });
}

// One conjugate-gradient iteration of every problem in the batch (parity =
// iteration number mod 2 selects the slot holding the current r.z).
static void pcg_iteration(const DAArgs& a, const double* mu, int batch, PCGWork& w, int parity, double tol2,
                          cudaStream_t s) {
  MGHierarchy* mg = w.mg;
  if (mg && mg->nlev > 0) {
    const MGGrid g = mg_grid(a, batch);
    MG_DISPATCH(a, pcg_spmv_mg, g, s, mg_dev(mg->lev[0], w), w);
    pcg_update_mg<<<g.grid, g.block, 0, s>>>(a.N, w, parity, tol2);
    mg_vcycle(*mg, w, batch, parity ^ 1, s);
    pcg_pupdate_mg<<<g.grid, g.block, 0, s>>>(a.N, w, parity, 0);
    return;
  }
  const dim3 grid(kPCGBlocks, batch);
  pcg_spmv_kernel<<<grid, kThreads, 0, s>>>(a, mu, w);
  pcg_reduce_kernel<<<batch, kThreads, 0, s>>>(w, 2, -1, -1);
  pcg_update_kernel<<<grid, kThreads, 0, s>>>(a, w, parity);
  pcg_reduce_kernel<<<batch, kThreads, 0, s>>>(w, parity ^ 1, 3, -1);
  pcg_pupdate_kernel<<<grid, kThreads, 0, s>>>(a, w, parity);
  pcg_mark_done_kernel<<<(batch + 127) / 128, 128, 0, s>>>(w, batch, tol2);
}

int pcg_solve(const DAArgs& a, const double* mu_in, int batch, const double* rhs, double* x, PCGWork& w,
              int max_iter, double tol, cudaStream_t s, cudaError_t* err) {
  const dim3 grid(kPCGBlocks, batch);
  const double tol2 = tol * tol;
  MGHierarchy* mg = w.mg;
  const bool multigrid = mg && mg->nlev > 0;
  cudaMemsetAsync(w.scal, 0, sizeof(double) * 8 * batch, s);
  const double* mu = w.mu;
  if (multigrid) {
    // level 0 of the hierarchy works on the PCG vectors (the V-cycle maps r to
    // z); the iterations read the levels' diagonals, built here from mu, so
    // that a captured chunk of them stays valid for every call
    MGLevel& L0 = mg->lev[0];
    L0.A = a;
    L0.d = w.b;
    L0.w = w.dinv;
    L0.b = w.r;
    L0.x = w.z;
    w.mg_x2 = L0.x2;
    mg_diag_kernel<<<mg_blocks(a.N, batch), kThreads, 0, s>>>(a, mu_in, mg->omega, L0.d, L0.w);
    const double* muf = mu_in;
    for (int l = 1; l < mg->nlev; ++l) {
      const DAArgs& f = mg->lev[l - 1].A;
      MGLevel& L = mg->lev[l];
      mg_coarsen_kernel<<<mg_blocks(L.A.N, batch), kThreads, 0, s>>>(f, L.A, muf, mg->omega, L.mu, L.d, L.w);
      muf = L.mu;
    }
    const MGGrid g = mg_grid(a, batch);
    pcg_init_mg<<<g.grid, g.block, 0, s>>>(a.N, rhs, w);
    mg_vcycle(*mg, w, batch, 0, s);
    pcg_pupdate_mg<<<g.grid, g.block, 0, s>>>(a.N, w, 0, 1);
  } else {
    copy_kernel<<<256, kThreads, 0, s>>>((long long)batch * a.N, mu_in, w.mu);
    pcg_init_kernel<<<grid, kThreads, 0, s>>>(a, mu, rhs, w);
    pcg_reduce_kernel<<<batch, kThreads, 0, s>>>(w, 0, 3, 4);
  }
  *err = cudaGetLastError();
  if (*err != cudaSuccess) return -1;
  // the host looks at the convergence flags after every chunk of iterations
  // (an even number, so that every chunk starts at parity 0)
  const int chunk = multigrid ? kPCGChunk : 4 * kPCGChunk;
  if (w.use_graphs && w.chunk_batch != batch) {
    if (w.chunk) cudaGraphExecDestroy(w.chunk);
    w.chunk = nullptr;
    w.chunk_batch = 0;
    if (!w.cap && (*err = cudaStreamCreateWithFlags(&w.cap, cudaStreamNonBlocking)) != cudaSuccess) return -1;
    if ((*err = cudaStreamBeginCapture(w.cap, cudaStreamCaptureModeThreadLocal)) != cudaSuccess) return -1;
    for (int k = 0; k < chunk; ++k) {
      pcg_iteration(a, mu, batch, w, k & 1, tol2, w.cap);
    }
    cudaGraph_t g = nullptr;
    *err = cudaStreamEndCapture(w.cap, &g);
    if (*err != cudaSuccess) return -1;
    *err = cudaGraphInstantiate(&w.chunk, g, 0);
    cudaGraphDestroy(g);
    if (*err != cudaSuccess) { w.chunk = nullptr; return -1; }
    w.chunk_batch = batch;
  }
  int it = 0;
  int used = -1;
  while (it < max_iter) {
    const int len = std::min(chunk, max_iter - it);
    if (w.use_graphs && len == chunk) {
      if ((*err = cudaGraphLaunch(w.chunk, s)) != cudaSuccess) return -1;
    } else {
      for (int k = 0; k < len; ++k) {
        pcg_iteration(a, mu, batch, w, k & 1, tol2, s);
      }
    }
    it += len;
    cudaMemcpyAsync(w.hostscal, w.scal, sizeof(double) * 8 * batch, cudaMemcpyDeviceToHost, s);
    cudaError_t e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) { *err = e; return -1; }
    bool all = true;
    for (int b = 0; b < batch; ++b) all = all && (w.hostscal[8 * b + 5] != 0.0);
    if (all) { used = it; break; }
  }
  copy_kernel<<<256, kThreads, 0, s>>>((long long)batch * a.N, w.x, x);
  *err = cudaGetLastError();
  return used;
}

__global__ void hadamard_kernel(long long n, double alpha, const double* u, const double* v, double* out) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = alpha * u[t] * v[t];
}

cudaError_t da_hadamard(int batch, int N, double alpha, const double* u, const double* v, double* out,
                        cudaStream_t s) {
  hadamard_kernel<<<512, kThreads, 0, s>>>((long long)batch * N, alpha, u, v, out);
  return cudaGetLastError();
}

template <typename T>
__global__ void heating_kernel(long long n, const double* a1, const double* b1, const double* a2, const double* b2,
                               T* out) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x) {
    double v = a1[t] * b1[t];
    if (a2) v += a2[t] * b2[t];
    out[t] = (T)v;
  }
}

template <typename T>
cudaError_t da_heating_T(int batch, int N, const double* a1, const double* b1, const double* a2, const double* b2,
                         T* out, cudaStream_t s) {
  heating_kernel<T><<<512, kThreads, 0, s>>>((long long)batch * N, a1, b1, a2, b2, out);
  return cudaGetLastError();
}

template <typename T>
__global__ void adjoint_out_kernel(long long n, const double* phi, const T* hbar, const double* ht, double* g) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    g[t] = phi[t] * ((double)hbar[t] + ht[t]);
}

template <typename T>
cudaError_t da_adjoint_out(int batch, int N, const double* phi, const T* hbar, const double* ht, double* g,
                           cudaStream_t s) {
  adjoint_out_kernel<T><<<512, kThreads, 0, s>>>((long long)batch * N, phi, hbar, ht, g);
  return cudaGetLastError();
}

template <typename T>
__global__ void to_double_kernel(long long n, const T* in, double* out) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = (double)in[t];
}

template <typename T>
cudaError_t T_to_double(long long n, const T* in, double* out, cudaStream_t s) {
  to_double_kernel<T><<<512, kThreads, 0, s>>>(n, in, out);
  return cudaGetLastError();
}

template <typename T>
__global__ void adjoint_rhs_kernel(long long n, double scale, const double* mu, const T* hbar, double* out) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    out[t] = scale * mu[t] * (double)hbar[t];
}

template <typename T>
cudaError_t da_adjoint_rhs(int batch, int N, double scale, const double* mu, const T* hbar, double* out,
                           cudaStream_t s) {
  adjoint_rhs_kernel<T><<<512, kThreads, 0, s>>>((long long)batch * N, scale, mu, hbar, out);
  return cudaGetLastError();
}

// ---- derivatives in kappa --------------------------------------------------
// d/da of the harmonic mean 2ab/(a+b)
__device__ __forceinline__ double dharmonic(double a, double b) { return 2.0 * b * b / ((a + b) * (a + b)); }

// Per cell c: the faces to its neighbours (axis, direction) and its boundary
// sides.  mode 0: out = delta-b - delta-A phi for dkappa (gather form: the
// face (c, nb) changes its coefficient by hf (dh(k_c, k_nb) dk_c +
// dh(k_nb, k_c) dk_nb) and contributes -delta-t (phi_c - phi_nb); a boundary
// side s adds 2 q dk_c (I_s - gamma phi_c) with q = d/dk of k h^(d-1)/(gamma h
// + k)).  mode 1: out = the kappa gradient sum over faces of
// -dh(k_c, k_nb) hf (phi_c - phi_nb)(psi_c - psi_nb) plus 2 q (I_s - gamma
// phi_c) psi_c per boundary side.
__global__ void kappa_deriv_kernel(DAArgs a, const double* kappa, const double* phi, const double* v, unsigned mask,
                                   double* out, int mode, double scale) {
  const long long o = (long long)blockIdx.y * a.N;
  const double hf = (a.dim == 3) ? a.h : 1.0;
  const double hb = (a.dim == 3) ? a.h * a.h : a.h;
  const int sy = a.n0, sz = a.n0 * a.n1;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < a.N; g += gridDim.x * blockDim.x) {
    const int i = g % a.n0, j = (g / a.n0) % a.n1, k = g / sz;
    const double kc = kappa[g], pc = phi[o + g], vc = v[o + g];
    double acc = 0.0;
    const int nbs[6] = {i > 0 ? g - 1 : -1, i < a.n0 - 1 ? g + 1 : -1, j > 0 ? g - sy : -1,
                        j < a.n1 - 1 ? g + sy : -1, (a.dim == 3 && k > 0) ? g - sz : -1,
                        (a.dim == 3 && k < a.n2 - 1) ? g + sz : -1};
    for (int f = 0; f < 6; ++f) {
      const int nb = nbs[f];
      if (nb < 0) continue;
      const double kn = kappa[nb];
      if (mode == 0) {
        const double dt = hf * (dharmonic(kc, kn) * vc + dharmonic(kn, kc) * v[o + nb]);
        acc -= dt * (pc - phi[o + nb]);
      } else {
        acc -= dharmonic(kc, kn) * hf * (pc - phi[o + nb]) * (vc - v[o + nb]);
      }
    }
    const double gh = a.gamma * a.h;
    const double q = gh * hb / ((gh + kc) * (gh + kc));
    const bool on[6] = {i == 0, i == a.n0 - 1, j == 0, j == a.n1 - 1, a.dim == 3 && k == 0,
                        a.dim == 3 && k == a.n2 - 1};
    for (int s = 0; s < 2 * a.dim; ++s) {
      if (!on[s]) continue;
      const double I = ((mask >> s) & 1u) ? 1.0 : 0.0;
      acc += 2.0 * q * (I - a.gamma * pc) * vc;
    }
    out[o + g] = scale * acc;
  }
}

cudaError_t da_kappa_source(const DAArgs& a, const double* kappa, int batch, const double* phi, const double* dkappa,
                            unsigned mask, double* out, cudaStream_t s) {
  kappa_deriv_kernel<<<dim3(128, batch), kThreads, 0, s>>>(a, kappa, phi, dkappa, mask, out, 0, 1.0);
  return cudaGetLastError();
}

cudaError_t da_kappa_grad(const DAArgs& a, const double* kappa, int batch, const double* phi, const double* psi,
                          unsigned mask, double scale, double* out, cudaStream_t s) {
  kappa_deriv_kernel<<<dim3(128, batch), kThreads, 0, s>>>(a, kappa, phi, psi, mask, out, 1, scale);
  return cudaGetLastError();
}

__global__ void axpy_kernel(long long n, double alpha, const double* x, double* y) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n; t += (long long)gridDim.x * blockDim.x)
    y[t] += alpha * x[t];
}

cudaError_t da_axpy(long long n, double alpha, const double* x, double* y, cudaStream_t s) {
  axpy_kernel<<<512, kThreads, 0, s>>>(n, alpha, x, y);
  return cudaGetLastError();
}

// Inner products in FP64: per thread a Neumaier-compensated running sum of
// the FP64 products, a fixed-order tree over the block, and a compensated
// sequential sum of the block partials.
__device__ __forceinline__ void neumaier(double& s, double& c, double v) {
  const double t = s + v;
  if (fabs(s) >= fabs(v)) c += (s - t) + v;
  else c += (v - t) + s;
  s = t;
}

template <typename T>
__global__ void dot_partial_kernel(long long len, const T* a, const T* b, double* partial) {
  const int bb = blockIdx.y;
  const T* x = a + (long long)bb * len;
  const T* y = b + (long long)bb * len;
  double s = 0, c = 0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < len; t += (long long)gridDim.x * blockDim.x)
    neumaier(s, c, (double)x[t] * (double)y[t]);
  block_sum3(s, c, 0.0, partial + ((long long)bb * kPartials + blockIdx.x) * 4);
}

__global__ void dot_final_kernel(const double* partial, double* out, int batch) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= batch) return;
  double s = 0, c = 0;
  for (int t = 0; t < kPartials; ++t) {
    neumaier(s, c, partial[((long long)b * kPartials + t) * 4]);
    neumaier(s, c, partial[((long long)b * kPartials + t) * 4 + 1]);
  }
  out[b] = s + c;
}

template <typename T>
cudaError_t dot_compensated(int batch, long long len, const T* a, const T* b, double* d_partial, double* d_out,
                            cudaStream_t s) {
  dot_partial_kernel<T><<<dim3(kPartials, batch), kThreads, 0, s>>>(len, a, b, d_partial);
  dot_final_kernel<<<(batch + 127) / 128, 128, 0, s>>>(d_partial, d_out, batch);
  return cudaGetLastError();
}

#define QPAT_DA_INST(T)                                                                                  \
  template cudaError_t da_heating_T<T>(int, int, const double*, const double*, const double*,           \
                                       const double*, T*, cudaStream_t);                                 \
  template cudaError_t da_adjoint_out<T>(int, int, const double*, const T*, const double*, double*,      \
                                         cudaStream_t);                                                  \
  template cudaError_t T_to_double<T>(long long, const T*, double*, cudaStream_t);                      \
  template cudaError_t da_adjoint_rhs<T>(int, int, double, const double*, const T*, double*, cudaStream_t); \
  template cudaError_t dot_compensated<T>(int, long long, const T*, const T*, double*, double*, cudaStream_t);
QPAT_DA_INST(float)
QPAT_DA_INST(double)

}  // namespace qpat
