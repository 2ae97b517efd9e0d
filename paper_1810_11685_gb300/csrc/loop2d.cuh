// The time loop of a small 2D FP32 grid as one kernel.
//
// One thread-block cluster holds one problem: CTA r of the cluster owns a
// block of row pairs and a block of column pairs (kx, -kx) for the whole
// loop, with its rows' state, its rows' medium and its columns' k-space
// symbols in shared memory.  The spectra are exchanged through L2 (the
// context's spectral buffer), with one cluster barrier between passes.  A
// grid of this size has too little work for a launch per pass: at 168^2 each
// of the six passes of a step took 4.4-5.5 us, nearly all of it launch, table
// loads and one warp's serial chain; here a pass takes 3.6 us (2.4 us at 56^2),
// bound by its chain of five barriers, the write-out before the cluster
// barrier (15% of the warps' time) and the load from L2 behind it.  Measured on
// GB300, forward + adjoint, launched passes against this: 168^2, one problem,
// 400 steps 25.8 -> 17.6 ms; 96^2, 200 steps 18.6 -> 5.8 ms; 120^2 x 4, Jacobian
// product over 400 steps 16.6 -> 7.4 ms; 150 x 210 lossless x 2 (runtime
// lengths), 200 steps 10.8 -> 8.3 ms.
//
// Layout.  Two real fields f0, f1 travel as one complex field f0 + i f1, so a
// row pass is one complex x-FFT in and one out per grid row with no split or
// merge, and the two rows of a pair run as one stream of packed FP32x2
// instructions.  A column pass holds the columns kx and -kx of it: with
// A(y) = Z(kx, y) and B(y) = conj Z(-kx, y), the forward y-FFTs give
// F0 = (A + B)/2 and F1 = (A - B)/(2i) at (kx, ky) in one thread, and the
// products G0, G1 return as U = G0 + i G1 and V = G0 - i G1, whose inverse
// transforms are the columns kx and (conjugated) -kx.  A and B are the two
// lanes of the packed stream.  A single field (the pressure) is packed as two
// rows p_j + i p_(j+1), which the column pass separates as it loads.
// Fields that share a transform are balanced by powers of two (PropArgs su to
// sa), so that neither's rounding drowns the other.
//
// Each transform is a Stockham FFT of three stages, with its length known at
// compile time for the square grids listed in loop2d.h and compile-time
// butterflies at runtime lengths for the others.  The first stage reads global memory, the
// last stage of the inverse, the pointwise update and the first stage of the
// forward transform share one set of registers (the forward plan is the
// inverse one reversed), and the last stage writes global memory.
#pragma once
#include "fft_reg.cuh"
#include "loop2d.h"
#include "pass_ops.cuh"

namespace qpat {

// Pass of one launch index (loop_pass).
struct LoopStep {
  int ph, n, flags;
};

// The passes of one step in order, one byte each.
constexpr unsigned long long loop_order(int p0, int p1, int p2, int p3, int p4 = 0, int p5 = 0) {
  const int p[6] = {p0, p1, p2, p3, p4, p5};
  unsigned long long v = 0;
  for (int k = 0; k < 6; ++k) v |= (unsigned long long)p[k] << (8 * k);
  return v;
}

// Pass g of a loop of nt samples.  Forward: g = n P + slot from n = -1 (P = 6,
// or 4 without absorption); adjoint: step k = g / P is n = nt - 2 - k.
template <bool ADJ, bool LL>
__host__ __device__ inline LoopStep loop_pass(int g, int nt) {
  constexpr int P = LL ? 4 : 6;
  constexpr unsigned long long order = ADJ ? (LL ? loop_order(A_R1L, A_C4, A_R5, A_C6)
                                                 : loop_order(A_R1, A_C2, A_R3, A_C4, A_R5, A_C6))
                                           : (LL ? loop_order(F_C1, F_R2, F_C2, F_R3L)
                                                 : loop_order(F_R1, F_C1, F_R2, F_C2, F_R3, F_C3));
  const int q = ADJ ? g / P : (g + P) / P - 1, slot = g - q * P;
  LoopStep s{(int)((order >> (8 * slot)) & 255), 0, 0};
  if (!ADJ) {
    s.n = q;
    if (s.ph == F_R1 && q == nt - 1) s.flags = kSkipOutput;
    if (s.ph == F_R3 || s.ph == F_R3L) s.flags = q == -1 ? (kSkipInput | kSource) : q == 0 ? kSource : 0;
  } else {
    const int n = nt - 2 - q;
    s.n = n + 1;                                                 // the sample p_(n+1)
    const int acc = n == 0 ? kAccWrite : n == -1 ? kAccAdd : 0, last = n == -1 ? kSkipOutput : 0;
    if (slot == 0 && n == nt - 2) s.flags = kSkipInput;
    if (slot == (LL ? 0 : 2)) s.flags |= acc | last;
  }
  return s;
}

__device__ __forceinline__ void cluster_arrive() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ int cluster_rank() {
  int r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

// Twiddles of one axis as the stages read them, W_L^(k r step) at r Ns + k
// (r from 1): mid and last stage of the order (q0, q1, q2), then of (q2, q1, q0).
struct LoopTw {
  const float2 *mid, *last, *mid2, *last2;
};
// What the stages of a pass share (one copy per thread, all uniform).
struct LoopCtx {
  int L, q0, q1, q2, mv;   // transform length, radices, lines of this CTA
  float4 *src, *dst;       // Stockham buffers
  int stride;              // line stride in 16-byte entries
  float2* spec;            // this problem's exchange buffer
  long long rs;            // its row stride
  int line0;               // first row pair / first column
  int nx;
};
// Quotients by a compile-time divisor D, or by d when D is 0.
template <int D>
struct LoopDiv {
  FastDiv f;
  __device__ __forceinline__ explicit LoopDiv(int d) : f(D ? 1 : d) {}
  __device__ __forceinline__ int div(int t) const { return D ? (int)((unsigned)t / (unsigned)(D ? D : 1)) : f.div(t); }
};

// First stage of a pass: what a line is and where its points are read.
enum LoopIn : int { kInRow2, kInRowHalf, kInCol2, kInCol1 };
// Last stage: where its points are written.
enum LoopOut : int { kOutRow2, kOutRow1, kOutCol2, kOutColHalf };

// Entry (row, column) of a problem's exchange buffer.
struct LoopCell {
  int row, col;
};
__host__ __device__ constexpr int loop_mirror(int kx, int nx) { return kx == 0 ? 0 : nx - kx; }
// Entries of point i of a line (a row pair or a column) in its first and last
// stage; `which` of the two that a packed pair takes.  The ranks of a cluster
// meet only between passes, so a pass may write no entry that another rank reads
// in it: a line's writes stay within the rows (the columns) that belong to it.
// The packed pressure of rows 2 line, 2 line + 1 therefore lies in row 2 line,
// although half the rows would hold it.
__host__ __device__ constexpr LoopCell loop_in_cell(int kind, int line, int i, int which, int nx) {
  return kind == kInRow2      ? LoopCell{2 * line + which, i}
         : kind == kInRowHalf ? LoopCell{2 * line + which, 2 * i <= nx ? i : nx - i}
                              : LoopCell{kind == kInCol1 ? i & ~1 : i, which ? loop_mirror(line, nx) : line};
}
__host__ __device__ constexpr LoopCell loop_out_cell(int kind, int line, int i, int which, int nx) {
  return kind == kOutRow2   ? LoopCell{2 * line + which, i}
         : kind == kOutRow1 ? LoopCell{2 * line, i}
                            : LoopCell{i, which ? loop_mirror(line, nx) : line};
}
// Whether pass ph takes in, or leaves, one field.
__host__ __device__ constexpr bool loop_one_in(int ph) { return ph == F_C1 || ph == A_R1 || ph == A_R1L; }
__host__ __device__ constexpr bool loop_one_out(int ph) { return ph == F_R1 || ph == F_R3L || ph == A_C6; }
__host__ __device__ constexpr bool loop_is_row(int ph) { return ph < 10 || (ph >= 20 && ph < 30); }
// f(integral constant of the kind) for pass ph's first stage, and for its last.
template <int K>
using LoopKind = std::integral_constant<int, K>;
#pragma nv_exec_check_disable
template <bool ADJ, class F>
__host__ __device__ __forceinline__ void loop_with_in(int ph, F&& f) {
  if constexpr (!ADJ) {
    if (loop_is_row(ph)) f(LoopKind<kInRow2>{});
    else if (loop_one_in(ph)) f(LoopKind<kInCol1>{});
    else f(LoopKind<kInCol2>{});
  } else {
    if (!loop_is_row(ph)) f(LoopKind<kInCol2>{});
    else if (loop_one_in(ph)) f(LoopKind<kInRowHalf>{});
    else f(LoopKind<kInRow2>{});
  }
}
#pragma nv_exec_check_disable
template <bool ADJ, class F>
__host__ __device__ __forceinline__ void loop_with_out(int ph, F&& f) {
  if constexpr (!ADJ) {
    if (!loop_is_row(ph)) f(LoopKind<kOutCol2>{});
    else if (loop_one_out(ph)) f(LoopKind<kOutRow1>{});
    else f(LoopKind<kOutRow2>{});
  } else {
    if (loop_is_row(ph)) f(LoopKind<kOutRow2>{});
    else if (loop_one_out(ph)) f(LoopKind<kOutColHalf>{});
    else f(LoopKind<kOutCol2>{});
  }
}

// Entry i of a line: a packed pair (16 bytes) or one complex value (8 bytes).
__device__ __forceinline__ void put(float4* line, int i, P2 v) { line[i] = p2_bits(v); }
__device__ __forceinline__ void put(float4* line, int i, float2 v) { reinterpret_cast<float2*>(line)[i] = v; }
template <typename E>
__device__ __forceinline__ E get(const float4* line, int i) {
  if constexpr (std::is_same<E, P2>::value) return p2_from(line[i]);
  else return reinterpret_cast<const float2*>(line)[i];
}
// Operands j + r L/R of a stage of radix R into v, from the planes of a first
// stage of radix RF (PLANES) or a line in order.  R RF divides L, so that all
// operands of j are in plane j mod RF.
template <int LC, int R, bool PLANES, typename E>
__device__ __forceinline__ void gather_operands(const LoopCtx& c, const float4* line, int j, int RF, int pitch, E (&v)[R]) {
  const int L = LC ? LC : c.L, nb = L / R;
  if constexpr (PLANES) {
    const int q = LC ? j / RF : FastDiv(RF).div(j), step = nb / RF;
    const int a = (j - q * RF) * pitch + q;
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = get<E>(line, a + r * step);
  } else {
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = get<E>(line, j + r * nb);
  }
}

template <int KIND>
__device__ __forceinline__ auto load_point(const LoopCtx& c, int m, int i, int L) {
  const int line = c.line0 + m;
  auto at = [&](int which) {
    const LoopCell q = loop_in_cell(KIND, line, i, which, c.nx);
    return __ldcg(c.spec + (long long)q.row * c.rs + q.col);
  };
  if constexpr (KIND == kInRow2) {                               // conj of rows 2 line, 2 line + 1
    return pack2(cconj(at(0)), cconj(at(1)));
  } else if constexpr (KIND == kInRowHalf) {                     // conj(P + i Q) of two rows' half spectra
    float2 P = at(0), Q = at(1);
    if (i == 0 || 2 * i == L) { P.y = 0.f; Q.y = 0.f; }
    if (2 * i > L) { P.y = -P.y; Q.y = -Q.y; }
    return make_float2(P.x - Q.y, -(P.y + Q.x));
  } else if constexpr (KIND == kInCol2) {
    return pack2(at(0), cconj(at(1)));
  } else {                                                       // row i of a field packed two rows to a line
    const float2 Z = at(0), Zm = cconj(at(1));
    return (i & 1) ? cscale(cmul_mi(csub(Z, Zm)), 0.5f) : cscale(cadd(Z, Zm), 0.5f);
  }
}

template <int KIND, typename E>
__device__ __forceinline__ void store_point(const LoopCtx& c, int m, int i, E v) {
  const int line = c.line0 + m;
  auto put_at = [&](int which, float2 z) {
    const LoopCell q = loop_out_cell(KIND, line, i, which, c.nx);
    c.spec[(long long)q.row * c.rs + q.col] = z;
  };
  if constexpr (KIND == kOutRow2) {
    put_at(0, lane0(v));
    put_at(1, lane1(v));
  } else if constexpr (KIND == kOutRow1) {
    put_at(0, v);
  } else if constexpr (KIND == kOutCol2) {
    put_at(0, cconj(lane0(v)));
    if (loop_mirror(line, c.nx) != line) put_at(1, lane1(v));
  } else {
    put_at(0, cconj(v));
  }
}

constexpr bool in_pair(int kind) { return kind == kInRow2 || kind == kInCol2; }
constexpr bool out_pair(int kind) { return kind == kOutRow2 || kind == kOutCol2; }

// Stage with stride 1 from global memory into the planes of c.dst.  Rows:
// adjacent threads take adjacent points of a line; columns: adjacent lines
// (adjacent kx), so that either way a warp reads runs of the exchange buffer's
// rows.
template <int LC, int R, int KIND>
__device__ __forceinline__ void first_stage(const LoopCtx& c) {
  typedef typename std::conditional<in_pair(KIND), P2, float2>::type E;
  constexpr bool row = KIND == kInRow2 || KIND == kInRowHalf;
  const int L = LC ? LC : c.L, nb = L / R, tot = c.mv * nb, pitch = loop_pitch(nb);
  const LoopDiv<row ? LC / R : 0> by(row ? nb : (c.mv > 0 ? c.mv : 1));
  for (int t = threadIdx.x; t < tot; t += loop_threads(LC)) {
    const int q = by.div(t), rem = t - q * (row ? nb : c.mv);
    const int m = row ? q : rem, j = row ? rem : q;
    E v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = load_point<KIND>(c, m, j + r * nb, L);
    dft<R, LC != 0>(v);
    float4* line = c.dst + m * c.stride;
#pragma unroll
    for (int r = 0; r < R; ++r) put(line, j + r * pitch, v[r]);
  }
}

// Middle stage of radix R after a first stage of radix RF (stride Ns = RF),
// from the planes of c.src to lines in order in c.dst.
template <int LC, int R, typename E>
__device__ __forceinline__ void mid_stage(const LoopCtx& c, int RF, const float2* tw) {
  const int L = LC ? LC : c.L, nb = L / R, tot = c.mv * nb, pitch = loop_pitch(L / RF);
  const LoopDiv<LC / R> by_nb(nb);
  for (int t = threadIdx.x; t < tot; t += loop_threads(LC)) {
    const int m = by_nb.div(t), j = t - m * nb;
    const int q = LC ? j / RF : FastDiv(RF).div(j), k = j - q * RF;
    E v[R];
    gather_operands<LC, R, true>(c, c.src + m * c.stride, j, RF, pitch, v);
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[(r - 1) * RF + k]);
    dft<R, LC != 0>(v);
    float4* out = c.dst + m * c.stride;
    const int o = q * RF * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) put(out, o + r * RF, v[r]);
  }
}

// Last stage (stride L/R), c.src to global memory.
template <int LC, int R, int KIND>
__device__ __forceinline__ void last_stage(const LoopCtx& c, const float2* tw) {
  typedef typename std::conditional<out_pair(KIND), P2, float2>::type E;
  constexpr bool row = KIND == kOutRow2 || KIND == kOutRow1;
  const int L = LC ? LC : c.L, nb = L / R, tot = c.mv * nb;
  const LoopDiv<row ? LC / R : 0> by(row ? nb : (c.mv > 0 ? c.mv : 1));
  for (int t = threadIdx.x; t < tot; t += loop_threads(LC)) {
    const int q = by.div(t), rem = t - q * (row ? nb : c.mv);
    const int m = row ? q : rem, j = row ? rem : q;
    E v[R];
    gather_operands<LC, R, false>(c, c.src + m * c.stride, j, 0, 0, v);
#pragma unroll
    for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[(r - 1) * nb + j]);
    dft<R, LC != 0>(v);
#pragma unroll
    for (int r = 0; r < R; ++r) store_point<KIND>(c, m, j + r * nb, v[r]);
  }
}

// This CTA's share of the loop's data in shared memory.
struct LoopShared {
  float2 *vx, *vy, *rx, *ry, *pb, *sc;          // state of row pair m at m nx + i: (row j0, row j0 + 1)
  const float2 *Cc, *rho, *dx, *dy, *eta, *tau; // medium, the same layout
  const float *kap, *kp1, *kp2;                 // symbols of column m at m ny + ky
  const float2 *shp, *shm;                      // y shift factors [ny]
  const float *ax, *asx;                        // PML along x [nx]
  const float2 *ay, *asy;                       // PML of the row pairs [rp]
};

__device__ __forceinline__ bool not_finite(F2 v) { return !isfinite(v.v.x) || !isfinite(v.v.y); }

// Pointwise update of grid points (i, j0) and (i, j0 + 1), j0 = 2 (line0 + m),
// from the incoming fields f0, f1 (both rows in one packed pair each).
template <int PH>
__device__ __forceinline__ void loop_row_point(const LoopArgs& A, const LoopShared& S, const LoopCtx& c, int nx, int b,
                                               int m, int i, int flags, F2 f0, F2 f1, F2& o0, F2& o1, bool& bad) {
  const PropArgs<float>& a = A.a;
  const int p = m * nx + i, j0 = 2 * (c.line0 + m);
  o0 = F2(0.f);
  o1 = F2(0.f);
  if constexpr (PH == F_R1 || PH == F_R3L) {
    F2 pr;
    if constexpr (PH == F_R1) {                                  // eq. num-p
      const F2 r = F2(S.rx[p]) + F2(S.ry[p]);
      const F2 t = r - F2(S.eta[p]) * f0;
      pr = F2(S.Cc[p]) * F2(t + F2(S.tau[p]) * f1);
    }
    if constexpr (PH == F_R1) {
      float* pb = a.pbuf + (long long)b * a.gstride + (long long)j0 * nx + i;
      pb[0] = pr.v.x;
      pb[nx] = pr.v.y;
      bad |= not_finite(pr);
      o0 = pr;
    }
  }
  if constexpr (PH == F_R2) {                                    // eq. num-vel
    const F2 sx(S.asx[i]), sy(S.asy[m]);
    const F2 vx = sx * F2(sx * F2(S.vx[p]) - F2(S.dx[p]) * f0);
    const F2 vy = sy * F2(sy * F2(S.vy[p]) - F2(S.dy[p]) * f1);
    S.vx[p] = vx.v;
    S.vy[p] = vy.v;
    o0 = vx;
    o1 = vy;
  }
  if constexpr (PH == F_R3 || PH == F_R3L) {                     // eq. num-rho, source of eq. s1
    F2 q(0.f);
    if ((flags & kSource) && i >= a.pml && i < a.pml + a.n0) {
      const float* p0 = a.io->p0 + (long long)b * a.n0 * a.n1 + (i - a.pml);
      const float2 C = S.Cc[p];
      const int y0 = j0 - a.pml, y1 = y0 + 1;
      q = F2(y0 >= 0 && y0 < a.n1 ? p0[(long long)y0 * a.n0] / (4.f * C.x) : 0.f,
             y1 >= 0 && y1 < a.n1 ? p0[(long long)y1 * a.n0] / (4.f * C.y) : 0.f);
    }
    const F2 ax(S.ax[i]), ay(S.ay[m]), r0(S.rho[p]);
    const F2 dr = F2(r0 * F2(a.dt));
    F2 rx(S.rx[p]), ry(S.ry[p]);
    if (PH == F_R3 || !(flags & kRebuild)) {
      rx = q + ax * F2(ax * rx - dr * f0);
      ry = q + ay * F2(ay * ry - dr * f1);
      S.rx[p] = rx.v;
      S.ry[p] = ry.v;
    }
    if constexpr (PH == F_R3) {
      o0 = rx + ry;
      const F2 ux = F2(ax * r0), uy = F2(ay * r0);
      o1 = F2(F2(A.a.su) * F2(F2(ux * f0) + uy * f1));
    } else {
      const F2 pr = F2(F2(S.Cc[p]) * (rx + ry));
      float* pb = a.pbuf + (long long)b * a.gstride + (long long)j0 * nx + i;
      pb[0] = pr.v.x;
      pb[nx] = pr.v.y;
      bad |= not_finite(pr);
      o0 = pr;
    }
  }
  if constexpr (PH == A_R1) {                                    // transpose of num-m and num-p
    const F2 Cp = F2(F2(S.Cc[p]) * (f0 + F2(S.sc[p])));
    S.pb[p] = Cp.v;
    o0 = F2(F2(S.eta[p]) * Cp);
    o1 = F2(F2(S.tau[p]) * Cp);
  }
  if constexpr (PH == A_R1L || PH == A_R3) {                     // transpose of num-rho and of the source
    F2 rpart, ya(0.f);
    if constexpr (PH == A_R1L) rpart = F2(F2(S.Cc[p]) * (f0 + F2(S.sc[p])));
    else {
      rpart = F2(S.pb[p]) - f0;
      ya = F2(f1 * F2(A.a.sa));                                    
    }
    const F2 ax(S.ax[i]), ay(S.ay[m]), r0(S.rho[p]);
    const F2 rtx = F2(S.rx[p]) + rpart, rty = F2(S.ry[p]) + rpart;
    o0 = F2(F2(r0 * ax) * F2(ya - F2(a.dt) * rtx));
    o1 = F2(F2(r0 * ay) * F2(ya - F2(a.dt) * rty));
    S.rx[p] = F2(F2(ax * ax) * rtx).v;
    S.ry[p] = F2(F2(ay * ay) * rty).v;
    const F2 sum = rtx + rty;
    bad |= not_finite(sum);
    if ((flags & (kAccWrite | kAccAdd)) && i >= a.pml && i < a.pml + a.n0) {
      float* dst = a.io->p0adj + (long long)b * a.n0 * a.n1 + (i - a.pml);
      const float2 C = S.Cc[p];
      const float val[2] = {sum.v.x / (4.f * C.x), sum.v.y / (4.f * C.y)};
#pragma unroll
      for (int rr = 0; rr < 2; ++rr) {
        const int y = j0 + rr - a.pml;
        if (y < 0 || y >= a.n1) continue;
        float* d = dst + (long long)y * a.n0;
        if (flags & kAccWrite) *d = val[rr];
        else *d += val[rr];
      }
    }
  }
  if constexpr (PH == A_R5) {                                    // transpose of num-vel
    const F2 sx(S.asx[i]), sy(S.asy[m]);
    const F2 vtx = F2(S.vx[p]) + f0, vty = F2(S.vy[p]) + f1;
    S.vx[p] = F2(F2(sx * sx) * vtx).v;
    S.vy[p] = F2(F2(sy * sy) * vty).v;
    o0 = F2(F2(sx * F2(S.dx[p])) * vtx);
    o1 = F2(F2(sy * F2(S.dy[p])) * vty);
  }
}

// Spectral products at (kx, ky) of column line m: F0, F1 in, G0, G1 out.
template <int PH>
__device__ __forceinline__ void loop_col_point(const LoopShared& S, int ny, int m, int ky, float2 sx, float2 F0,
                                               float2 F1, float2& G0, float2& G1) {
  const int t = m * ny + ky;
  if constexpr (PH == F_C3 || PH == A_C2) {
    G0 = cscale(F0, S.kp1[t]);
    G1 = cscale(F1, S.kp2[t]);
  } else {
    const float k = S.kap[t];
    const float2 sy = (PH == F_C1 || PH == A_C6) ? S.shp[ky] : S.shm[ky];
    if constexpr (PH == F_C1 || PH == F_C2) {
      G0 = cscale(cmul(sx, F0), k);
      G1 = cscale(cmul(sy, F1), k);
    } else if constexpr (PH == A_C4) {
      G0 = cscale(cmul(cconj(sx), F0), k);
      G1 = cscale(cmul(cconj(sy), F1), k);
    } else {
      G0 = cscale(cadd(cmul(cconj(sx), F0), cmul(cconj(sy), F1)), -k);
      G1 = G0;
    }
  }
}

// Last stage of the first transform, the update, and the first stage of the
// second transform (both of radix R), c.src to c.dst.
template <int LC, int R, int PH>
__device__ __forceinline__ void point_stage(const LoopArgs& A, const LoopShared& S, const LoopCtx& c, const float2* tw,
                                            int b, int flags, bool& bad) {
  constexpr bool row = loop_is_row(PH), in1 = loop_one_in(PH), out1 = loop_one_out(PH);
  typedef typename std::conditional<in1, float2, P2>::type Ei;
  typedef typename std::conditional<out1, float2, P2>::type Eo;
  const int L = LC ? LC : c.L, nb = L / R, tot = c.mv * nb, pitch = loop_pitch(nb);
  const int nx = LC ? LC : A.a.nx, ny = LC ? LC : A.a.ny;
  const LoopDiv<LC / R> by_nb(nb);
  for (int t = threadIdx.x; t < tot; t += loop_threads(LC)) {
    const int m = by_nb.div(t), j = t - m * nb;
    Ei v[R];
    if (flags & kSkipInput) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (in1) v[r] = make_float2(0.f, 0.f);
        else v[r] = P2{F2(0.f), F2(0.f)};
      }
    } else {
      gather_operands<LC, R, false>(c, c.src + m * c.stride, j, 0, 0, v);
#pragma unroll
      for (int r = 1; r < R; ++r) v[r] = cmul(v[r], tw[(r - 1) * nb + j]);
      dft<R, LC != 0>(v);
    }
    Eo o[R];
    if constexpr (row) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        // v = FFT(conj Z) = conj(f0 + i f1), or conj of the two rows of one field
        F2 f0, f1(0.f), o0, o1;
        if constexpr (in1) f0 = F2(v[r].x, -v[r].y);
        else { f0 = v[r].x; f1 = -v[r].y; }
        loop_row_point<PH>(A, S, c, nx, b, m, j + r * nb, flags, f0, f1, o0, o1, bad);
        if constexpr (out1) o[r] = o0.v;
        else o[r] = P2{o0, o1};
      }
    } else {
      const int kx = c.line0 + m;
      const float2 sx = (PH == F_C1 || PH == A_C6) ? A.a.shxp[kx] : A.a.shxm[kx];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        float2 F0, F1, G0, G1;
        if constexpr (in1) {
          F0 = v[r];
          F1 = F0;
        } else {
          const float2 X = lane0(v[r]), Y = lane1(v[r]);
          F0 = cscale(cadd(X, Y), 0.5f);
          F1 = cscale(cmul_mi(csub(X, Y)), 0.5f);
        }
        loop_col_point<PH>(S, ny, m, j + r * nb, sx, F0, F1, G0, G1);
        if constexpr (out1) o[r] = cconj(G0);
        else o[r] = pack2(make_float2(G0.x - G1.y, -(G0.y + G1.x)), make_float2(G0.x + G1.y, G1.x - G0.y));
      }
    }
    if (!(flags & kSkipOutput)) {
      dft<R, LC != 0>(o);
      float4* out = c.dst + m * c.stride;
#pragma unroll
      for (int r = 0; r < R; ++r) put(out, j + r * pitch, o[r]);
    }
  }
}

// The stages with the axis' radices: compile-time for LC, by switch for
// runtime lengths.
template <int LC, int KIND>
__device__ __forceinline__ void first_any(const LoopCtx& c) {
  if constexpr (LC) {
    first_stage<LC, loop_axis(LC).q[0], KIND>(c);
  } else {
    switch (c.q0) {
      case 3: first_stage<0, 3, KIND>(c); break;
      case 4: first_stage<0, 4, KIND>(c); break;
      case 5: first_stage<0, 5, KIND>(c); break;
      case 6: first_stage<0, 6, KIND>(c); break;
      case 7: first_stage<0, 7, KIND>(c); break;
      default: first_stage<0, 8, KIND>(c); break;
    }
  }
}
template <int LC, int KIND>
__device__ __forceinline__ void last_any(const LoopCtx& c, const float2* tw) {
  if constexpr (LC) {
    last_stage<LC, loop_axis(LC).q[0], KIND>(c, tw);
  } else {
    switch (c.q0) {
      case 3: last_stage<0, 3, KIND>(c, tw); break;
      case 4: last_stage<0, 4, KIND>(c, tw); break;
      case 5: last_stage<0, 5, KIND>(c, tw); break;
      case 6: last_stage<0, 6, KIND>(c, tw); break;
      case 7: last_stage<0, 7, KIND>(c, tw); break;
      default: last_stage<0, 8, KIND>(c, tw); break;
    }
  }
}
// Middle stage after a first stage of radix q0 (FWD) or q2.
template <int LC, typename E, bool FWD>
__device__ __forceinline__ void mid_any(const LoopCtx& c, const float2* tw) {
  if constexpr (LC) {
    mid_stage<LC, loop_axis(LC).q[1], E>(c, loop_axis(LC).q[FWD ? 0 : 2], tw);
  } else {
    const int RF = FWD ? c.q0 : c.q2;
    switch (c.q1) {
      case 2: mid_stage<0, 2, E>(c, RF, tw); break;
      case 3: mid_stage<0, 3, E>(c, RF, tw); break;
      case 4: mid_stage<0, 4, E>(c, RF, tw); break;
      case 5: mid_stage<0, 5, E>(c, RF, tw); break;
      case 6: mid_stage<0, 6, E>(c, RF, tw); break;
      case 7: mid_stage<0, 7, E>(c, RF, tw); break;
      default: mid_stage<0, 8, E>(c, RF, tw); break;
    }
  }
}
template <int LC, int PH>
__device__ __forceinline__ void point_any(const LoopArgs& A, const LoopShared& S, const LoopCtx& c, const float2* tw,
                                          int b, int flags, bool& bad) {
  if constexpr (LC) {
    point_stage<LC, loop_axis(LC).q[2], PH>(A, S, c, tw, b, flags, bad);
  } else {
    switch (c.q2) {
      case 4: point_stage<0, 4, PH>(A, S, c, tw, b, flags, bad); break;
      case 5: point_stage<0, 5, PH>(A, S, c, tw, b, flags, bad); break;
      case 6: point_stage<0, 6, PH>(A, S, c, tw, b, flags, bad); break;
      case 7: point_stage<0, 7, PH>(A, S, c, tw, b, flags, bad); break;
      default: point_stage<0, 8, PH>(A, S, c, tw, b, flags, bad); break;
    }
  }
}

// Stage twiddles of one axis into shared memory at t (loop_ntw entries), from
// the context's table W_L^m.
__device__ __forceinline__ LoopTw loop_twiddles(const LoopAxis& ax, const float2* w, float2* t, int nth) {
  auto stage = [&](int Ns, int R) {
    const int step = ax.L / (Ns * R);
    for (int u = threadIdx.x; u < Ns * (R - 1); u += nth) {
      const int r = u / Ns + 1, k = u - (r - 1) * Ns;
      t[u] = w[k * r * step];
    }
    const float2* at = t;
    t += Ns * (R - 1);
    return at;
  };
  LoopTw o;
  o.mid = stage(ax.q[0], ax.q[1]);
  o.last = stage(ax.q[0] * ax.q[1], ax.q[2]);
  o.mid2 = stage(ax.q[2], ax.q[1]);
  o.last2 = stage(ax.q[2] * ax.q[1], ax.q[0]);
  return o;
}

template <bool ADJ, bool LL, int LC>
__global__ void __launch_bounds__(loop_threads(LC), 1) loop2d_kernel(const __grid_constant__ LoopArgs A) {
  constexpr int NT = loop_threads(LC);
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const PropArgs<float>& a = A.a;
  const int nx = LC ? LC : a.nx, ny = LC ? LC : a.ny, tid = threadIdx.x;
  int nc;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(nc));
  const int rank = cluster_rank(), b = blockIdx.x / nc;
  const LoopLayout lay = loop_layout(A.x, A.y, A.rp, A.cp, A.stride, ADJ, LL);
  float* sm = reinterpret_cast<float*>(smem_raw);
  const int M = A.rp > A.cp ? A.rp : A.cp;
  float4* bufA = reinterpret_cast<float4*>(sm);
  float4* bufB = bufA + M * A.stride;
  float2* twp = reinterpret_cast<float2*>(sm + lay.tw);
  const LoopTw twx = loop_twiddles(A.x, a.twx, twp, NT),
               twy = loop_twiddles(A.y, a.twy, twp + loop_ntw(A.x), NT);
  float2* shp = twp + lay.ntw;
  float2* shm = shp + ny;
  float2* fld = reinterpret_cast<float2*>(sm + lay.fields);
  float* ktab = sm + lay.ktab;
  float* pax = sm + lay.pml;
  float* pasx = pax + nx;
  float2* pay = reinterpret_cast<float2*>(pasx + nx);
  float2* pasy = pay + A.rp;

  const int jp0 = rank * A.rp, npair = ny >> 1;
  const int rows = jp0 < npair ? (npair - jp0 < A.rp ? npair - jp0 : A.rp) : 0;
  const int kx0 = rank * A.cp;
  const int cols = kx0 < a.nxh ? (a.nxh - kx0 < A.cp ? a.nxh - kx0 : A.cp) : 0;
  const int per = A.rp * nx;                                     // points of one field

  LoopShared S;
  {
    float2* f = fld;
    auto take = [&]() { float2* r = f; f += per; return r; };
    S.vx = take(); S.vy = take(); S.rx = take(); S.ry = take();
    S.pb = ADJ && !LL ? take() : nullptr;
    S.sc = ADJ ? take() : nullptr;
    S.Cc = take(); S.rho = take(); S.dx = take(); S.dy = take();
    S.eta = LL ? nullptr : take();
    S.tau = LL ? nullptr : take();
    S.kap = ktab;
    S.kp1 = LL ? nullptr : ktab + A.cp * ny;
    S.kp2 = LL ? nullptr : ktab + 2 * A.cp * ny;
    S.shp = shp; S.shm = shm; S.ax = pax; S.asx = pasx; S.ay = pay; S.asy = pasy;
  }
  // state, medium, tables
  const float tau_scale = LL ? 1.f : ADJ ? A.a.st : A.a.sy;          
  for (int t = tid; t < rows * nx; t += NT) {
    const int m = t / nx, i = t - m * nx;
    const long long g = 2LL * (jp0 + m) * nx + i, gb = (long long)b * a.gstride + g;
    auto two = [&](const float* p, long long o) { return make_float2(p[o], p[o + nx]); };
    const float2 zero = make_float2(0.f, 0.f);
    S.vx[t] = A.load ? two(a.vx, gb) : zero;
    S.vy[t] = A.load ? two(a.vy, gb) : zero;
    S.rx[t] = A.load ? two(a.rx, gb) : zero;
    S.ry[t] = A.load ? two(a.ry, gb) : zero;
    if (ADJ) S.sc[t] = zero;
    const_cast<float2*>(S.Cc)[t] = two(a.Cc, g);
    const_cast<float2*>(S.rho)[t] = two(a.rho0, g);
    const_cast<float2*>(S.dx)[t] = two(a.dtrsx, g);
    const_cast<float2*>(S.dy)[t] = two(a.dtrsy, g);
    if (!LL) {
      const_cast<float2*>(S.eta)[t] = two(a.eta, g);
      const float2 ta = two(a.tau, g);
      const_cast<float2*>(S.tau)[t] = make_float2(ta.x * tau_scale, ta.y * tau_scale);
    }
  }
  // (the balance factors are powers of two: scaling a table by them is exact)
  const float kp2_scale = LL ? 1.f : ADJ ? 1.f / (A.a.st * A.a.sa) : 1.f / (A.a.su * A.a.sy);
  for (int t = tid; t < cols * ny; t += NT) {
    const int m = t / ny, ky = t - m * ny;
    const long long o = (long long)ky * a.nxh + kx0 + m;
    ktab[t] = a.kap[o];
    if (!LL) {
      ktab[A.cp * ny + t] = a.kp1[o];
      ktab[2 * A.cp * ny + t] = a.kp2[o] * kp2_scale;
    }
  }
  for (int t = tid; t < nx; t += NT) { pax[t] = a.ax[t]; pasx[t] = a.asx[t]; }
  for (int t = tid; t < ny; t += NT) { shp[t] = a.shyp[t]; shm[t] = a.shym[t]; }
  for (int t = tid; t < rows; t += NT) {
    const int j = 2 * (jp0 + t);
    pay[t] = make_float2(a.ay[j], a.ay[j + 1]);
    pasy[t] = make_float2(a.asy[j], a.asy[j + 1]);
  }
  __syncthreads();

  LoopCtx c;
  c.stride = A.stride;
  c.spec = a.spec + (long long)b * a.sstride;
  c.rs = 2LL * a.pitch;
  c.nx = nx;
  bool bad = false;
  const float* pall = a.pbuf + (long long)b * a.gstride;
  auto gather = [&](int n) {                                     // eq. num-m over the cluster's threads
    float* dn = a.io->data + ((long long)b * a.nt + n) * a.ns;
    for (int s = rank * NT + tid; s < a.ns; s += nc * NT) {
      float acc = 0.f;
#pragma unroll
      for (int q = 0; q < 4; ++q) acc += a.sw[4 * s + q] * __ldcg(pall + a.sidx[4 * s + q]);
      dn[s] = acc;
    }
  };

  // grid points of this CTA's rows that sensors touch
  const int pt0 = ADJ && rows > 0 ? a.rowptr[2 * jp0] : 0, pt1 = ADJ && rows > 0 ? a.rowptr[2 * (jp0 + rows)] : 0;

  cluster_arrive();
  for (int g = A.g0; g < A.g1; ++g) {
    const LoopStep st = loop_pass<ADJ, LL>(g, A.nt);
    const int ph = st.ph, flags = !ADJ && LL && A.rebuild && g == A.g0 ? kSkipInput | kRebuild : st.flags;
    const bool row = loop_is_row(ph);
    const LoopAxis& ax = row ? A.x : A.y;
    c.L = ax.L;
    c.q0 = ax.q[0];
    c.q1 = ax.q[1];
    c.q2 = ax.q[2];
    c.mv = row ? rows : cols;
    c.line0 = row ? jp0 : kx0;
    LoopTw tw;
    tw.mid = row ? twx.mid : twy.mid;
    tw.last = row ? twx.last : twy.last;
    tw.mid2 = row ? twx.mid2 : twy.mid2;
    tw.last2 = row ? twx.last2 : twy.last2;
    // M^T w_n on this CTA's rows (the same points in every step, zero elsewhere), before the wait
    if (ADJ && (ph == A_R1 || ph == A_R1L)) {
      const float* wn = a.io->w + ((long long)b * a.nt + st.n) * a.ns;
      float* sc = reinterpret_cast<float*>(S.sc);
      for (int q = pt0 + tid; q < pt1; q += NT) {
        float acc = 0.f;
        for (int e = a.pent[q]; e < a.pent[q + 1]; ++e) acc += a.ew[e] * wn[a.esens[e]];
        const int j = a.prow[q] - 2 * jp0;
        sc[2 * ((j >> 1) * nx + a.pcol[q]) + (j & 1)] = acc;
      }
    }
    cluster_wait();
    if (!ADJ && ph == F_C1) gather(st.n);
    float4 *p0 = bufA, *p1 = bufB;
    const bool in1 = loop_one_in(ph), out1 = loop_one_out(ph);
    if (!(flags & kSkipInput)) {
      c.dst = p0;
      loop_with_in<ADJ>(ph, [&](auto kind) { first_any<LC, decltype(kind)::value>(c); });
      __syncthreads();
      c.src = p0;
      c.dst = p1;
      if (in1) mid_any<LC, float2, true>(c, tw.mid);
      else mid_any<LC, P2, true>(c, tw.mid);
      __syncthreads();
      float4* t = p0; p0 = p1; p1 = t;
    } else {
      __syncthreads();                                           // the scatter above, before the update reads it
    }
    c.src = p0;
    c.dst = p1;
    if constexpr (!ADJ && !LL) {
      switch (ph) {
        case F_R1: point_any<LC, F_R1>(A, S, c, tw.last, b, flags, bad); break;
        case F_R2: point_any<LC, F_R2>(A, S, c, tw.last, b, flags, bad); break;
        case F_R3: point_any<LC, F_R3>(A, S, c, tw.last, b, flags, bad); break;
        case F_C1: point_any<LC, F_C1>(A, S, c, tw.last, b, flags, bad); break;
        case F_C2: point_any<LC, F_C2>(A, S, c, tw.last, b, flags, bad); break;
        default: point_any<LC, F_C3>(A, S, c, tw.last, b, flags, bad); break;
      }
    } else if constexpr (!ADJ) {
      switch (ph) {
        case F_R2: point_any<LC, F_R2>(A, S, c, tw.last, b, flags, bad); break;
        case F_R3L: point_any<LC, F_R3L>(A, S, c, tw.last, b, flags, bad); break;
        case F_C1: point_any<LC, F_C1>(A, S, c, tw.last, b, flags, bad); break;
        default: point_any<LC, F_C2>(A, S, c, tw.last, b, flags, bad); break;
      }
    } else if constexpr (!LL) {
      switch (ph) {
        case A_R1: point_any<LC, A_R1>(A, S, c, tw.last, b, flags, bad); break;
        case A_R3: point_any<LC, A_R3>(A, S, c, tw.last, b, flags, bad); break;
        case A_R5: point_any<LC, A_R5>(A, S, c, tw.last, b, flags, bad); break;
        case A_C2: point_any<LC, A_C2>(A, S, c, tw.last, b, flags, bad); break;
        case A_C4: point_any<LC, A_C4>(A, S, c, tw.last, b, flags, bad); break;
        default: point_any<LC, A_C6>(A, S, c, tw.last, b, flags, bad); break;
      }
    } else {
      switch (ph) {
        case A_R1L: point_any<LC, A_R1L>(A, S, c, tw.last, b, flags, bad); break;
        case A_R5: point_any<LC, A_R5>(A, S, c, tw.last, b, flags, bad); break;
        case A_C4: point_any<LC, A_C4>(A, S, c, tw.last, b, flags, bad); break;
        default: point_any<LC, A_C6>(A, S, c, tw.last, b, flags, bad); break;
      }
    }
    if (!(flags & kSkipOutput)) {
      __syncthreads();
      c.src = p1;
      c.dst = p0;
      if (out1) mid_any<LC, float2, false>(c, tw.mid2);
      else mid_any<LC, P2, false>(c, tw.mid2);
      __syncthreads();
      float4* t = p0; p0 = p1; p1 = t;
      c.src = p1;
      loop_with_out<ADJ>(ph, [&](auto kind) { last_any<LC, decltype(kind)::value>(c, tw.last2); });
    }
    cluster_arrive();
  }
  cluster_wait();
  if (!ADJ && A.gather_last) gather(A.nt - 1);
  if (A.save) {
    for (int t = tid; t < rows * nx; t += NT) {
      const int m = t / nx, i = t - m * nx;
      const long long gb = (long long)b * a.gstride + 2LL * (jp0 + m) * nx + i;
      auto two = [&](float* p, float2 v) { p[gb] = v.x; p[gb + nx] = v.y; };
      two(a.vx, S.vx[t]);
      two(a.vy, S.vy[t]);
      two(a.rx, S.rx[t]);
      two(a.ry, S.ry[t]);
    }
  }
  if (__syncthreads_or(bad) && tid == 0) atomicOr(a.err, 1);
}

// Clusters of nc CTAs resident at once (nc = 0: only set the attributes); 0 if
// they do not fit.
template <bool ADJ, bool LL, int LC>
int loop_occupancy_one(int nc, size_t smem) {
  if (smem > 227 * 1024) return 0;
  if (cudaFuncSetAttribute(loop2d_kernel<ADJ, LL, LC>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) !=
          cudaSuccess ||
      cudaFuncSetAttribute(loop2d_kernel<ADJ, LL, LC>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
          cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (nc == 0) return 1;
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(nc);
  cfg.blockDim = dim3(loop_threads(LC));
  cfg.dynamicSmemBytes = smem;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, loop2d_kernel<ADJ, LL, LC>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

template <bool ADJ, bool LL, int LC>
cudaError_t loop_launch_one(const LoopArgs& A, int nc, int batch, size_t smem, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = nc;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.gridDim = dim3(nc * batch);
  cfg.blockDim = dim3(loop_threads(LC));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, loop2d_kernel<ADJ, LL, LC>, A);
}

// The four kernels of extent L (QPAT_LOOP_INST), or for runtime lengths one of
// them per translation unit (QPAT_LOOP_INST0).
#define QPAT_LOOP_INST(L)                                                                              \
  template <>                                                                                          \
  cudaError_t loop_launch_len<L>(const LoopArgs& A, int adj, int ll, int nc, int batch, size_t smem,   \
                                 cudaStream_t s) {                                                     \
    if (adj)                                                                                           \
      return ll ? loop_launch_one<true, true, L>(A, nc, batch, smem, s)                                \
                : loop_launch_one<true, false, L>(A, nc, batch, smem, s);                              \
    return ll ? loop_launch_one<false, true, L>(A, nc, batch, smem, s)                                 \
              : loop_launch_one<false, false, L>(A, nc, batch, smem, s);                               \
  }                                                                                                    \
  template <>                                                                                          \
  int loop_occupancy_len<L>(int adj, int ll, int nc, size_t smem) {                                    \
    if (adj)                                                                                           \
      return ll ? loop_occupancy_one<true, true, L>(nc, smem) : loop_occupancy_one<true, false, L>(nc, smem); \
    return ll ? loop_occupancy_one<false, true, L>(nc, smem) : loop_occupancy_one<false, false, L>(nc, smem); \
  }
// Extent L without absorption only: with it the loop's data of a rank of sixteen
// is above the 227 KB of shared memory a CTA may use (loop_layout; 244 KB at 224).
#define QPAT_LOOP_INST_LOSSLESS(L)                                                                     \
  template <>                                                                                          \
  cudaError_t loop_launch_len<L>(const LoopArgs& A, int adj, int ll, int nc, int batch, size_t smem,   \
                                 cudaStream_t s) {                                                     \
    if (!ll) return cudaErrorInvalidValue;                                                             \
    return adj ? loop_launch_one<true, true, L>(A, nc, batch, smem, s)                                 \
               : loop_launch_one<false, true, L>(A, nc, batch, smem, s);                               \
  }                                                                                                    \
  template <>                                                                                          \
  int loop_occupancy_len<L>(int adj, int ll, int nc, size_t smem) {                                    \
    if (!ll) return 0;                                                                                 \
    return adj ? loop_occupancy_one<true, true, L>(nc, smem) : loop_occupancy_one<false, true, L>(nc, smem); \
  }
#define QPAT_LOOP_INST0(ADJ, LL)                                                                       \
  template int loop_occupancy_one<ADJ, LL, 0>(int, size_t);                                            \
  template cudaError_t loop_launch_one<ADJ, LL, 0>(const LoopArgs&, int, int, size_t, cudaStream_t);

}  // namespace qpat
