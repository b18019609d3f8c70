// Economy QR of the tall sketch S = C_k W^{(k)} (Algorithm 4) on GB300.
//
// Householder QR is a chain of rank-1 updates and would run on one SM at the
// FP64 rate of a single SM (~8 GFLOP/s on GB300). Cholesky QR instead spends
// almost all of its flops in two SM-parallel steps (the Gram S^T S, and
// S R^{-1} as a forward substitution with half a warp per row of S); only the
// c x c Cholesky factorization runs in one block. A pass is
//     G = S^T S,  R^T R = G (+ shift),  S <- S R^{-1}
// and passes repeat until G = I to working accuracy (Cholesky QR2 needs two
// passes for cond(S) < ~1e8). When the unshifted factorization breaks down
// (cond(S) >~ 1e8, or exactly dependent columns as in Y ⊙ Y or exact
// low-rank products), the pass uses the shift s = 11 (m c + c (c + 1)) u tr(G)
// of shifted Cholesky QR (Fukaya, Kannan, Nakatsukasa, Yamamoto, Yanagisawa,
// SIAM J. Sci. Comput. 2020); each shifted pass lifts the smallest singular
// values towards 1, so later passes converge. A column that is exactly zero
// stays zero (its Gram row and column vanish), which leaves a partial
// isometry whose zero columns carry nothing into the next core.
//
// An S of exactly lower rank than c (a raw TT representation, a sketch of an
// exact low-rank product) has null directions at the rounding level, ~u ||S||.
// Each shifted pass multiplies them by about 1/sqrt(s / ||S||^2), i.e. by 1e4
// to 1e6 for the sizes here, so they need four shifted passes to reach unit
// size and then one or two plain ones: six passes in all. Stopping earlier
// leaves Q far from orthonormal, and the projection Q Q^T C of the callers
// then loses about 1e-9 of C.
//
// A pass whose G is I to first order (the usual second one) needs no
// factorization (gram_load).
//
// Launch forms, the same passes:
//  * grid (qr_fused_kernel<., false>): all passes in one cooperative launch, one
//    block per SM, each block owning a contiguous slice of the rows of S. Grid
//    barriers separate the Gram partial sums, their reduction and, where one is
//    needed, the factorization (block 0); a converged QR stops at once, so no
//    launch and no no-op pass follows the convergence test. Used on calls whose
//    stream runs alone (single recompressions, rounding);
//  * cluster (qr_fused_kernel<., true>): the same in up to 8 blocks of one
//    cluster with its hardware barrier (~1200 clocks with the fence, 3000 to 4000
//    for the grid's), for sizes that 8 SMs finish in less than the grid barriers
//    take; any stream;
//  * launch per step: per pass the Gram shares, their sum, the
//    factorization and the apply, all passes launched unconditionally (fixed
//    launch sequence); a device flag set by the convergence test turns the
//    remaining launches into no-ops. Used by the batched entry points, whose
//    many streams would serialize on whole-GPU cooperative grids.
// All run the same device code on the same row partition, so they give
// bitwise the same Q; all are capturable in a CUDA graph.
//
// Bound: FP64 at 2 lanes per SM and clock for the Gram matrix and the apply from
// m c^2 ~ 1e7 on (c = 90: 82% of the time), barriers and the pivot chain below.
// Measured (us, Gaussian S, two passes; with a one-column factorization in both,
// a row per warp and no cluster form in parentheses): 50 x 5 20 (33), 96 x 12 26
// (38), 256 x 32 48 (60), 64 x 64 111 (206), 600 x 30 48 (56), 1600 x 50 78 (97),
// 5760 x 90 265 (314).
#include <algorithm>
#include <cmath>
#include <cstdlib>
#include <cstring>
#include "hatt_internal.cuh"
#include "rcp.cuh"

namespace hatt {
namespace {

__device__ int g_qr_health = 0;   // kHealthNonfinite / kHealthBreakdown bits
// The word a factorization notes them in: the caller's (set_health_word) or ours.
__device__ __forceinline__ int *health_word(int *word) { return word != nullptr ? word : &g_qr_health; }

constexpr int kPasses = 6;
constexpr int kCholThreads = 256;
constexpr int kTrsmThreads = 256;

// 1/sqrt(x) for finite x > 0: range reduction x = m 2^e with e even, an FP32
// seed for m, then two Newton-Raphson steps y <- y (3 - m y^2) / 2 in FP64
// (each squares the relative error: 2^-23 -> 2^-46 -> below FP64 rounding).
// A handful of dependent FP64 multiply-adds instead of the long FP64 sqrt and
// divide sequences, which sit on the Cholesky critical path once per column.
__device__ __forceinline__ double rsqrt_newton(double x) {
  int e;
  double m = frexp(x, &e);                 // m in [0.5, 1)
  if (e & 1) { m *= 2.0; e -= 1; }         // m in [0.5, 2), e even
  double y = (double)rsqrtf((float)m);
  y = y * fma(-0.5 * m, y * y, 1.5);
  y = y * fma(-0.5 * m, y * y, 1.5);
  return ldexp(y, -e / 2);
}

// 1/sqrt(x) for x in [1e-30, 1e30] (a pivot pre-scaled by an even power of
// two): the FP32 seed and the same two Newton-Raphson steps as rsqrt_newton,
// without its range reduction. On GB300 a dependent FP64 instruction costs
// ~64 clocks and frexp / ldexp are long sequences: measured 1447 clocks for
// rsqrt_newton against ~450 for this, on the critical path of every column.
__device__ __forceinline__ double rsqrt_scaled(double x) {
  const double h = -0.5 * x;
  double y = (double)rsqrtf((float)x);
  y = y * fma(h, y * y, 1.5);
  y = y * fma(h, y * y, 1.5);
  return y;
}

// Thresholds on the largest deviation of G from I, as the bit patterns of
// doubles (integer order equals numeric order for non-negative values, which
// keeps the comparisons off the FP64 unit).
struct QrTol {
  long long orth;                        // 8 c u: nothing to apply
  long long linear;                      // sqrt(u / c): a factor to first order is exact to u
  long long last;                        // 0.1 / c: the pass that applies is the last
};

// Flag words (zero at the start of every QR):
//   flags[0] done:      no further pass is needed (read at the start of every
//                       later pass of the launch-per-step form)
//   flags[1] skip_apply: the S <- S R^{-1} step of this pass is a no-op
//   flags[2] passes applied, flags[3] shifted passes (diagnostics)
//   flags[4] grid-barrier arrivals, flags[5] abort (grid form only)

enum { kQrFactor = 0, kQrOrthonormal = 1, kQrLinear = 2, kQrNonfinite = 3 };

// Shared state of a block that holds G.
struct QrShared {
  long long red[2][kCholThreads / 32];
  double rinv[kMaxSmall + 1];              // 1 / pivot, scaled
  double piv[kMaxSmall + 1];               // pivot, scaled
  double row[2][2][kMaxSmall];             // a panel's two rows (double buffer) ...
  double srow[2][2][kMaxSmall];            // ... and the same over their pivots
  unsigned char zero[kMaxSmall + 1];       // column j of S is exactly zero
};

// G from global memory (through L2: other blocks of the same launch wrote it)
// into shared memory (leading dimension c + 1), and what the pass does with it.
// The convergence test is absolute on purpose: S of any scale (HaTT sketches of
// long chains reach 1e-20 and below) is never mistaken for a converged basis.
// Exactly zero columns do not count (they stay zero through every pass).
//
// kQrLinear: R = I + H, H = E's strict upper part plus half its diagonal, has
// R^T R = G + H^T H, and the entries of H^T H stay below c max|E|^2 <= u. So the
// unit factor is G's strict upper part and 1 / R_jj = 1 - E_jj / 2: no
// factorization. This is the usual second pass (max|E| ~ u cond(S)^2 after the
// first), and every block takes it from its own copy of G.
__device__ __forceinline__ int gram_load(const double *Gg, int c, const QrTol &tol, double *G,
                                         QrShared &sh, long long &dev, long long &dmax) {
  const int ld = c + 1, n = c * c;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  dev = 0;
  dmax = 0;
  int bad = 0;
  // entry e = i c + j of thread tid: (i, j) advanced by (di, dj) per step of
  // kCholThreads entries, with a carry, instead of a division per entry
  const int di = kCholThreads / c, dj = kCholThreads - (kCholThreads / c) * c;
  int i = tid / c, j = tid - (tid / c) * c;
  constexpr int kLoads = 16;             // in flight per thread
  for (int e0 = tid; e0 < n; e0 += kLoads * kCholThreads) {
    double v[kLoads];
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      const int e = e0 + q * kCholThreads;
      v[q] = e < n ? __ldcg(Gg + e) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < kLoads; ++q) {
      if (e0 + q * kCholThreads >= n) break;
      long long bits = __double_as_longlong(v[q]) & 0x7fffffffffffffffLL;
      bad |= bits >= 0x7ff0000000000000LL;                   // Inf or NaN
      G[i * ld + j] = v[q];
      if (i == j) {
        sh.zero[i] = bits == 0;
        dmax = max(dmax, bits);
        bits = bits == 0 ? 0 : __double_as_longlong(v[q] - 1.0) & 0x7fffffffffffffffLL;
      }
      dev = max(dev, bits);
      i += di;
      j += dj;
      if (j >= c) {
        j -= c;
        ++i;
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) {
    dev = max(dev, __shfl_xor_sync(0xffffffffu, dev, o));
    dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
  }
  if (lane == 0) {
    sh.red[0][warp] = dev;
    sh.red[1][warp] = dmax;
  }
  if (__syncthreads_or(bad)) return kQrNonfinite;
  for (int w = 0; w < kCholThreads / 32; ++w) {
    dev = max(dev, sh.red[0][w]);
    dmax = max(dmax, sh.red[1][w]);
  }
  return dev <= tol.orth ? kQrOrthonormal : dev <= tol.linear ? kQrLinear : kQrFactor;
}

// y_j = 1 / R_jj of a kQrLinear pass.
__device__ __forceinline__ void linear_scale(const double *G, int c, const QrShared &sh, double *y) {
  for (int i = threadIdx.x; i < c; i += kCholThreads)
    y[i] = sh.zero[i] ? 1.0 : fma(-0.5, G[i * (c + 1) + i], 1.5);
}

// x 2^k for finite x on the bits (below the normal range: 0); the diagonal of
// the scaled matrix is of order 1 at most, such entries do not matter there.
__device__ __forceinline__ double scale_exp(double x, int k) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  return e == 0 || e + k <= 0 ? 0.0 : __longlong_as_double(b + ((long long)k << 52));
}

// Panel p of the factorization by warp 0: rows j = 2 p and j + 1 of the
// triangle, brought up to date with panel p - 1, their pivots and the rows over
// the pivots (row j of U~, published at once). A row and a pivot cost a chain of
// dependent FP64 instructions (~64 clocks each on GB300), one after the other:
// here both pivots come from the 2 x 2 block at once, its determinant
// d = g00 g11 - g01^2 (error u g00 g11, i.e. u g11 on the pivot d / g00, as in
// g11 - g01^2 / g00) and two reciprocals side by side.
// An exactly zero column of S (zero Gram diagonal) gets pivot 1, which leaves
// Q_j = 0 and couples nothing; sending it to the shifted attempt instead would
// make every pass shifted and leave ||Q^T Q - I|| at the shift (~1e-11) on an
// otherwise benign S. A pivot not safely positive fails the unshifted attempt;
// in the shifted attempt it sets the breakdown bit and is clamped so that
// nothing divides by zero.
// L: slots of 32 columns from the pivots' one to the end, a compile-time
// constant: branches around each slot cost more than the slot's arithmetic.
template <int L>
__device__ __forceinline__ void chol_panel(const double *G, int c, int p, QrShared &sh, long long floor_bits,
                                           double clamp, int attempt, double *Ut_g, int *health) {
  const int ld = c + 1, lane = threadIdx.x & 31;
  const int i0 = 2 * p, i1 = i0 + 1, i1c = min(i1, c - 1);
  const int l0 = (i0 & ~31) + lane;
  const double *r0 = sh.row[(p & 1) ^ 1][0], *r1 = sh.row[(p & 1) ^ 1][1];
  const double *w0 = sh.srow[(p & 1) ^ 1][0], *w1 = sh.srow[(p & 1) ^ 1][1];
  const double a00 = w0[i0], a01 = w1[i0], a10 = w0[i1c], a11 = w1[i1c];
  double x[L], z[L];
#pragma unroll
  for (int s = 0; s < L; ++s) {
    const int l = min(l0 + 32 * s, c - 1);
    const double b0 = r0[l], b1 = r1[l];
    x[s] = fma(-a01, b1, fma(-a00, b0, G[i0 * ld + l]));
    z[s] = fma(-a11, b1, fma(-a10, b0, G[i1c * ld + l]));
  }
  const double g00 = __shfl_sync(0xffffffffu, x[0], i0 & 31);
  const double g01 = __shfl_sync(0xffffffffu, x[0], i1 & 31);
  const double g11 = __shfl_sync(0xffffffffu, z[0], i1 & 31);
  const bool one = i1 >= c, z0 = sh.zero[i0], z1 = one || sh.zero[i1];
  const double det = fma(g00, g11, -(g01 * g01));
  double p0 = g00, p1, y0, y1;
  if (!z0 && !z1 && rcp_range(g00) && rcp_range(det)) {
    y0 = rcp_seeded(g00);
    const double yd = rcp_seeded(det);
    y1 = g00 * yd;
    p1 = det * y0;
  } else {
    bool fail = !z0 && __double_as_longlong(p0) <= floor_bits;
    if (z0) p0 = 1.0;
    else if (fail) p0 = clamp;
    y0 = 1.0 / p0;
    p1 = fma(-(g01 * y0), g01, g11);
    if (z1) p1 = 1.0;
    else if (__double_as_longlong(p1) <= floor_bits) {
      fail = true;
      p1 = clamp;
    }
    y1 = 1.0 / p1;
    if (fail && attempt != 0 && lane == 0) atomicOr(health_word(health), kHealthBreakdown);
  }
  const double l01 = g01 * y0;
  double *row = sh.row[p & 1][0], *srow = sh.srow[p & 1][0];
#pragma unroll
  for (int s = 0; s < L; ++s) {
    const int l = l0 + 32 * s;
    const double xs = x[s] * y0;
    const double zn = fma(-l01, x[s], z[s]), zs = zn * y1;
    if (l < c) {
      row[l] = x[s];
      srow[l] = xs;
      row[kMaxSmall + l] = zn;
      srow[kMaxSmall + l] = zs;
      Ut_g[i0 * c + l] = xs;             // entries up to the diagonal are not read
      if (!one) Ut_g[i1 * c + l] = zs;
    }
  }
  if (lane == 0) {
    sh.piv[i0] = p0;
    sh.piv[i1] = one ? 1.0 : p1;
  }
}

// One block: the Cholesky factor R of G (shifted if the plain factorization
// breaks down), published as the strict upper part of U~ = D^{-1} R and
// y = diag(D^{-1}), D = diag(R). G is in shared memory (gram_load).
//
// Right-looking, two columns per step, with look-ahead: while warps 1..7 apply
// panel p to the rows below (two multiply-adds per entry; the rows over the
// pivots are the multipliers, so none is formed twice), warp 0 brings the next
// two rows up to date and forms their panel: one barrier and one pivot chain
// per two columns. Bound: that chain (1000 clocks per column up to c = 32, 1250
// at c = 50, where the rows below compete for the FP64 unit; one column per
// step: 1500 and 1640), at c = 90 the FP64 unit.
// G is factorized scaled by 2^-2k, which puts the largest diagonal near 1
// (exact: a power of two), so the pivots that matter and their products are
// normal FP32 numbers; the floor and the clamp are scaled alike.
__device__ __forceinline__ void chol_factor(double *G, const double *Gg, double *Ut_g, double *y_g, int c,
                                            int m, long long dmax_bits, QrShared &sh, int *flags,
                                            int *health) {
  const int ld = c + 1;
  const int tid = threadIdx.x, warp = tid >> 5;
  const double dmax = __longlong_as_double(dmax_bits);
  const int be = (int)(dmax_bits >> 52);
  int ex = 0;
  if (be > 0) ex = be - 1022;                 // dmax = f 2^ex, f in [0.5, 1)
  else if (dmax > 0.0) frexp(dmax, &ex);
  const int k = ex / 2;
  const bool plain = be > 0 && k > -500 && k < 500;
  const double sc = plain ? __longlong_as_double((long long)(1023 - 2 * k) << 52) : ldexp(1.0, -2 * k);
  const double unsc = plain ? __longlong_as_double((long long)(1023 - k) << 52) : ldexp(1.0, -k);
  if (k != 0)
    for (int e = tid; e < c * ld; e += kCholThreads) {
      // (the padding column of a row is scaled along with it)
      G[e] = plain ? scale_exp(G[e], -2 * k) : G[e] * sc;
    }
  const double u = 1.1102230246251565e-16;
  const int np = (c + 1) / 2;
  for (int attempt = 0; attempt < 2; ++attempt) {
    double shift = 0.0;
    if (attempt == 1) {
      double trace = 0.0;
      for (int i = tid & 31; i < c; i += 32) trace += __ldcg(Gg + i * c + i);
      for (int o = 16; o > 0; o >>= 1) trace += __shfl_xor_sync(0xffffffffu, trace, o);
      shift = 11.0 * ((double)m * c + (double)c * (c + 1)) * u * trace;
      if (!(shift > 0.0)) shift = 1e-300;
      for (int e = tid; e < c * c; e += kCholThreads) {
        const int i = e / c, j = e % c;
        G[i * ld + j] = (__ldcg(Gg + e) + (i == j ? shift : 0.0)) * sc;
      }
      if (tid == 0) flags[3] += 1;
    }
    // no panel before the first
    for (int e = tid; e < 2 * kMaxSmall; e += kCholThreads) sh.row[1][0][e] = sh.srow[1][0][e] = 0.0;
    __syncthreads();
    // a non-negative floor as a bit pattern: a pivot passes if its bits, as a
    // signed integer, are larger (a negative one's never are)
    const long long floor_bits = (attempt == 0) ? __double_as_longlong((double)c * u * dmax * sc) : 0;
    const double clamp = fmax(shift, 1e-300) * sc;
    auto panel = [&](int p) {
      switch ((c + 31) / 32 - (p >> 4)) {
        case 1: chol_panel<1>(G, c, p, sh, floor_bits, clamp, attempt, Ut_g, health); break;
        case 2: chol_panel<2>(G, c, p, sh, floor_bits, clamp, attempt, Ut_g, health); break;
        case 3: chol_panel<3>(G, c, p, sh, floor_bits, clamp, attempt, Ut_g, health); break;
        default: chol_panel<4>(G, c, p, sh, floor_bits, clamp, attempt, Ut_g, health); break;
      }
    };
    if (warp == 0) panel(0);
    __syncthreads();
    bool failed = false;
    for (int p = 0; p < np; ++p) {
      // pivots from before the last barrier: all threads leave at the same panel
      // (a failed one is at most the floor, also after the clamp)
      if (attempt == 0 && min(__double_as_longlong(sh.piv[2 * p]), __double_as_longlong(sh.piv[2 * p + 1])) <=
                              floor_bits) {
        failed = true;
        break;
      }
      if (warp == 0) {
        if (p + 1 < np) panel(p + 1);
      } else {                            // 28 rows x 8 columns of threads
        const int bt = tid - 32, bx = bt & 7, by = bt >> 3;
        const double *r0 = sh.row[p & 1][0], *r1 = sh.row[p & 1][1];
        for (int i = 2 * p + 4 + by; i < c; i += 28) {
          const double a0 = sh.srow[p & 1][0][i], a1 = sh.srow[p & 1][1][i];
          for (int l = i + bx; l < c; l += 8) G[i * ld + l] = fma(-a1, r1[l], fma(-a0, r0[l], G[i * ld + l]));
        }
      }
      __syncthreads();
    }
    if (!failed) break;
    __syncthreads();                      // all reads of G and the pivots done before the retry
  }
  for (int i = tid; i < c; i += kCholThreads) {
    double yi = 1.0;                      // 1 / R_ii (1 for an exactly zero column)
    if (!sh.zero[i]) {                    // the pivot is sc R_ii^2, sc = unsc^2
      const double ps = sh.piv[i];
      yi = ((ps >= 1e-30 && ps <= 1e30) ? rsqrt_scaled(ps) : rsqrt_newton(ps)) * unsc;
    }
    y_g[i] = yi;
  }
}

// Launch per step: what the pass does, and its factor.
__global__ void __launch_bounds__(kCholThreads)
chol_inv_kernel(const double *Gg, double *Ut_g, double *y_g, int c, int m, QrTol tol, int *flags, int *health) {
  pdl_enter();
  if (flags[0]) {
    if (threadIdx.x == 0) flags[1] = 1;
    return;
  }
  extern __shared__ double sm[];
  __shared__ QrShared sh;
  long long dev, dmax;
  const int what = gram_load(Gg, c, tol, sm, sh, dev, dmax);
  if (what == kQrNonfinite || what == kQrOrthonormal) {
    if (threadIdx.x == 0) {
      if (what == kQrNonfinite) atomicOr(health_word(health), kHealthNonfinite);
      flags[0] = 1;
      flags[1] = 1;
    }
    return;
  }
  if (what == kQrLinear) {
    linear_scale(sm, c, sh, y_g);
    for (int e = threadIdx.x; e < c * c; e += kCholThreads) Ut_g[e] = sm[e + e / c];
  } else {
    chol_factor(sm, Gg, Ut_g, y_g, c, m, dmax, sh, flags, health);
  }
  if (threadIdx.x == 0) {
    flags[1] = 0;
    flags[2] += 1;
    if (dev <= tol.last) flags[0] = 1;
  }
}

// Q = S R^{-1} = (S U~^{-1}) D^{-1}, half a warp per row, in place. The unit
// diagonal keeps divisions out of the chain; the final scaling by y = D^{-1}
// is one multiply per entry. U~ (Us) and y (ys) in shared memory.
// A row takes half a warp (lane t of it: columns t, t + 16, ...): a step updates
// the slots of 16 columns from its own on, and the FP64 unit, which bounds the
// solve, spends 16 clocks on a warp-wide instruction however few lanes it has
// (a row per warp: 60% more instructions at c = 50, 17% at c = 90). The slots a
// step touches are chosen by warp-uniform loop bounds.
template <int NS>
__device__ __forceinline__ void apply_half(double *S, long long ldS, int c, const double *Us, int ld,
                                           const double *ys, int r0, int r1, int h, int halves) {
  const int hl = threadIdx.x & 15;
  for (int rw = r0 + (h & ~1); rw < r1; rw += halves) {        // the same for both halves of a warp
    const int r = rw + (h & 1);
    double *row = S + (long long)r * ldS;
    double x[NS];
#pragma unroll
    for (int s = 0; s < NS; ++s) x[s] = r < r1 && hl + 16 * s < c ? row[hl + 16 * s] : 0.0;
#pragma unroll
    for (int s0 = 0; s0 < NS; ++s0) {
      const int lend = min(c, 16 * (s0 + 1));
      for (int l = 16 * s0; l < lend; ++l) {
        const double xl = __shfl_sync(0xffffffffu, x[s0], l & 15, 16);
        const double *u = Us + l * ld;
#pragma unroll
        for (int s = s0; s < NS; ++s) {
          const int col = hl + 16 * s;
          if (col > l && col < c) x[s] = fma(-xl, u[col], x[s]);
        }
      }
    }
#pragma unroll
    for (int s = 0; s < NS; ++s)
      if (r < r1 && hl + 16 * s < c) row[hl + 16 * s] = x[s] * ys[hl + 16 * s];
  }
}

// Rows r0 + h, r0 + h + halves, ... < r1 of half-warp h (of `halves`).
__device__ __forceinline__ void apply_rows(double *S, long long ldS, int c, const double *Us, int ld,
                                           const double *ys, int r0, int r1, int h, int halves) {
  switch ((c + 15) / 16) {
    case 1: apply_half<1>(S, ldS, c, Us, ld, ys, r0, r1, h, halves); break;
    case 2: apply_half<2>(S, ldS, c, Us, ld, ys, r0, r1, h, halves); break;
    case 3: apply_half<3>(S, ldS, c, Us, ld, ys, r0, r1, h, halves); break;
    case 4: apply_half<4>(S, ldS, c, Us, ld, ys, r0, r1, h, halves); break;
    case 5: apply_half<5>(S, ldS, c, Us, ld, ys, r0, r1, h, halves); break;
    case 6: apply_half<6>(S, ldS, c, Us, ld, ys, r0, r1, h, halves); break;
    case 7: apply_half<7>(S, ldS, c, Us, ld, ys, r0, r1, h, halves); break;
    default: apply_half<8>(S, ldS, c, Us, ld, ys, r0, r1, h, halves); break;
  }
}

__global__ void __launch_bounds__(kTrsmThreads)
trsm_rows_kernel(double *S, int m, int c, long long ldS, const double *Ut, const double *y,
                 const int *flags) {
  pdl_enter();
  if (flags[1]) return;
  extern __shared__ double sm[];
  double *Us = sm;                       // c x c
  double *ys = sm + c * c;               // c
  for (int e = threadIdx.x; e < c * c; e += kTrsmThreads) Us[e] = Ut[e];
  for (int e = threadIdx.x; e < c; e += kTrsmThreads) ys[e] = y[e];
  __syncthreads();
  const int halves = kTrsmThreads / 16;
  apply_rows(S, ldS, c, Us, c, ys, 0, m, blockIdx.x * halves + (threadIdx.x >> 4), gridDim.x * halves);
}

// ------------------------------------------------------- the Gram matrix ---
// G = S^T S from per-block shares: block b of nb sums the rows [b p, b p + p)
// of S, p = ceil(m / nb), into the upper triangle (i <= j, c (c + 1) / 2
// entries) of its own share, and a warp then sums each entry over the nb
// shares. Both forms of the QR run these same device functions with the
// same nb (qr_blocks), so they compute bitwise the same G, and the same QR.
constexpr int kQrMaxBlocks = 160;       // >= the SMs of the device (152 on GB300)
constexpr int kQrRowTile = 16;          // rows of S staged per Gram step
constexpr int kQrMinRows = 4;           // rows per block at least (small m: fewer blocks)
// Gram entries a thread owns at most: c <= 64 and c <= kMaxSmall (two
// instantiations, so the common small case carries a quarter of the slots)
constexpr int kQrSlots64 = (64 * 65 / 2 + kCholThreads - 1) / kCholThreads;
constexpr int kQrMaxSlots = (kMaxSmall * (kMaxSmall + 1) / 2 + kCholThreads - 1) / kCholThreads;
constexpr int kClusterBlocks = 8;        // blocks of the cluster form at most (a power of two)
constexpr long long kClusterFma = 1 << 15;    // m c (c + 1) / 2 up to which it is taken
constexpr long long kQrSpinCap = 1LL << 21;   // polls of one barrier wait (seconds)

// Row i and column j >= i of entry o of the upper triangle of a c x c matrix
// stored by rows (row i starts at i c - i (i - 1) / 2): the root of the
// quadratic, then exact integer correction.
__device__ __forceinline__ void upper_index(int o, int c, int &i, int &j) {
  const float b = 2.0f * c + 1.0f;
  i = (int)((b - sqrtf(b * b - 8.0f * o)) * 0.5f);
  i = max(0, min(i, c - 1));
  while (i + 1 < c && (i + 1) * c - (i + 1) * i / 2 <= o) ++i;
  while (i > 0 && i * c - i * (i - 1) / 2 > o) --i;
  j = i + (o - (i * c - i * (i - 1) / 2));
}

// Entries of a share this thread sums: t, t + 256, ... (nq of them, packed
// as i << 8 | j); nqw = the most any lane of the warp has (lane 0's). Each
// warp runs the multiply-adds of nqw slots by warp-uniform branches, as the
// GEMM does (a predicated-off DFMA costs as much as a full one).
template <int MAXQ>
struct GramSlots {
  int pk[MAXQ];
  int nq, nqw;
};

template <int MAXQ>
__device__ __forceinline__ void gram_slots(int c, GramSlots<MAXQ> &g) {
  const int tid = threadIdx.x;
  const int T = c * (c + 1) / 2;
  g.nq = max(0, (T - tid + kCholThreads - 1) / kCholThreads);
  g.nqw = __shfl_sync(0xffffffffu, g.nq, 0);
#pragma unroll
  for (int q = 0; q < MAXQ; ++q) {
    int i = 0, j = 0;
    if (q < g.nq) upper_index(tid + kCholThreads * q, c, i, j);
    g.pk[q] = (i << 8) | j;
  }
}

// This block's share of the rows [r0, r1) of S, into mine (T entries); sm
// holds kQrRowTile rows of S. S is read through L2 (another block of the
// fused launch may have written it).
template <int MAXQ>
__device__ __forceinline__ void gram_share(const double *S, long long ldS, int c, int r0, int r1,
                                           const GramSlots<MAXQ> &g, double *mine, double *sm) {
  const int tid = threadIdx.x;
  double acc[MAXQ];
#pragma unroll
  for (int q = 0; q < MAXQ; ++q) acc[q] = 0.0;
  for (int rt = r0; rt < r1; rt += kQrRowTile) {
    const int rows = min(kQrRowTile, r1 - rt);
    for (int e = tid; e < rows * c; e += kCholThreads) {
      const int rr = e / c;
      sm[e] = __ldcg(S + (long long)(rt + rr) * ldS + (e - rr * c));
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < MAXQ; ++q) {
      if (q < g.nqw) {
        const double *a = sm + (g.pk[q] >> 8), *b = sm + (g.pk[q] & 255);
        double v = acc[q];
#pragma unroll 4
        for (int r = 0; r < rows; ++r) v = fma(a[r * c], b[r * c], v);
        acc[q] = v;
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int q = 0; q < MAXQ; ++q)
    if (q < g.nq) mine[tid + kCholThreads * q] = acc[q];
}

// Entries of G summed over the nb shares by warp w of `warps`: eight lanes per
// entry, four entries per warp (a warp per entry spends 10 FP64 instructions on
// each, this 5.5), all loads in flight, then a fixed order.
__device__ __forceinline__ void gram_entries(const double *part, int nb, int c, int w, int warps, double *G) {
  const int lane = threadIdx.x & 31, l8 = lane & 7;
  const int T = c * (c + 1) / 2;
  constexpr int kPer = kQrMaxBlocks / 8;
  for (int tw = 4 * w; tw < T; tw += 4 * warps) {
    const int t = tw + (lane >> 3);
    const bool in = t < T;
    double sh[kPer];
#pragma unroll
    for (int k = 0; k < kPer; ++k)
      sh[k] = in && l8 + 8 * k < nb ? __ldcg(part + (long long)(l8 + 8 * k) * T + t) : 0.0;
    int i = 0, j = 0;
    if (in) upper_index(t, c, i, j);
    double v = 0.0, v1 = 0.0;
#pragma unroll
    for (int k = 0; k < kPer; k += 2)
      if (8 * k < nb) {                   // the same for the whole warp
        v += sh[k];
        v1 += sh[k + 1];
      }
    v += v1;
    for (int o = 4; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (in && l8 == 0) {
      G[i * c + j] = v;
      G[j * c + i] = v;
    }
  }
}

// Launch per step: the shares (nb blocks), then their sum. Both do nothing
// once the QR has converged.
template <int MAXQ>
__global__ void __launch_bounds__(kCholThreads)
gram_share_kernel(const double *S, long long ldS, int m, int c, double *part, const int *flags) {
  pdl_enter();
  if (flags[0]) return;
  extern __shared__ double sm[];
  GramSlots<MAXQ> g;
  gram_slots(c, g);
  const int per = (m + gridDim.x - 1) / gridDim.x;
  const int r0 = min(m, (int)blockIdx.x * per), r1 = min(m, r0 + per);
  gram_share(S, ldS, c, r0, r1, g, part + (long long)blockIdx.x * (c * (c + 1) / 2), sm);
}

__global__ void __launch_bounds__(kCholThreads)
gram_sum_kernel(const double *part, int nb, int c, double *G, const int *flags) {
  pdl_enter();
  if (flags[0]) return;
  const int warps = gridDim.x * (kCholThreads / 32);
  gram_entries(part, nb, c, blockIdx.x * (kCholThreads / 32) + (threadIdx.x >> 5), warps, G);
}

// ------------------------------------------------------------ fused form ---
// Grid barrier of the fused QR (cooperative launch: every block is resident).
// Arrivals count up in bar[0] (zero at the start of the QR); the e-th barrier
// waits for e * gridDim.x of them. A wait gives up after spin_cap polls,
// sets the timeout health bit and bar[1] (abort), and every block that sees
// bar[1] gives up too: the QR then stops with S partly processed, and the
// device status reports the timeout. Returns false in that case.
__device__ __forceinline__ bool grid_barrier(int *bar, int &epoch, long long spin_cap) {
  ++epoch;
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&bar[0], 1);
    const int target = epoch * (int)gridDim.x;
    volatile int *vb = bar;
    long long polls = 0;
    while (vb[0] < target) {
      if (vb[1] != 0) { ok = 0; break; }
      if (++polls > spin_cap) {
        atomicOr(&g_qr_health, kHealthTimeout);
        atomicExch(&bar[1], 1);
        ok = 0;
        break;
      }
      __nanosleep(32);
    }
    __threadfence();
  }
  return __syncthreads_and(ok) != 0;
}

// All passes of one Cholesky QR of S (m x c, leading dimension ldS) in one
// launch of nb blocks, block b owning the rows [b p, b p + p) of S. A pass:
//   1. the block's Gram share -> part[b];
//   2. barrier; each warp sums entries of G over the shares (gram_entries);
//   3. barrier; every block loads G and takes the same decision (gram_load):
//      the QR ends (orthonormal, or G non-finite), or the factor follows from G
//      to first order, or block 0 factorizes (chol_factor) and a barrier follows;
//   4. R^{-1} applied to the block's own rows; if the pass was the last, the QR
//      ends here, else a barrier and the next pass.
// The passes, G, tests and factors are those of the launch-per-step form, bit
// for bit. CL: the blocks are one cluster, its hardware barrier takes the place
// of the grid barrier (flags then need no clearing).
template <int MAXQ, bool CL>
__global__ void __launch_bounds__(kCholThreads, 1)
qr_fused_kernel(double *S, int m, int c, long long ldS, double *G, double *Ut, double *y,
                double *part, QrTol tol, int *flags, int *health, long long spin_cap) {
  pdl_enter();
  extern __shared__ double sm[];
  __shared__ QrShared sh;
  double *ys = sm + c * (c + 1);
  const int tid = threadIdx.x, warp = tid >> 5;
  constexpr int kWarps = kCholThreads / 32;
  const int nb = gridDim.x, bid = blockIdx.x;
  const int per = (m + nb - 1) / nb;
  const int r0 = min(m, bid * per), r1 = min(m, r0 + per);
  const int T = c * (c + 1) / 2;
  GramSlots<MAXQ> g;
  gram_slots(c, g);
  int epoch = 0;
  if (CL && bid == 0 && tid == 0) flags[0] = flags[1] = flags[2] = flags[3] = 0;
  auto barrier = [&]() {
    if constexpr (CL) {
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
      return true;
    } else {
      return grid_barrier(flags + 4, epoch, spin_cap);
    }
  };
  for (int pass = 0; pass < kPasses; ++pass) {
    gram_share(S, ldS, c, r0, r1, g, part + (long long)bid * T, sm);
    if (!barrier()) return;
    gram_entries(part, nb, c, bid * kWarps + warp, nb * kWarps, G);
    if (!barrier()) return;
    long long dev, dmax;
    const int what = gram_load(G, c, tol, sm, sh, dev, dmax);
    const bool stop = what == kQrNonfinite || what == kQrOrthonormal, last = stop || dev <= tol.last;
    if (bid == 0 && tid == 0) {
      if (what == kQrNonfinite) atomicOr(health_word(health), kHealthNonfinite);
      flags[0] = last;
      flags[1] = stop;
      flags[2] += !stop;
    }
    if (stop) return;
    int ldu = c + 1;
    if (what == kQrLinear) {
      linear_scale(sm, c, sh, ys);
    } else {
      if (bid == 0) chol_factor(sm, G, Ut, y, c, m, dmax, sh, flags, health);
      if (!barrier()) return;
      ldu = c;
      for (int e = tid; e < c * c; e += kCholThreads) sm[e] = __ldcg(Ut + e);
      for (int e = tid; e < c; e += kCholThreads) ys[e] = __ldcg(y + e);
    }
    __syncthreads();
    apply_rows(S, ldS, c, sm, ldu, ys, r0, r1, tid >> 4, 2 * kWarps);
    if (last) return;
    if (!barrier()) return;
  }
}

// ------------------------------------------------- the one-column form ---
// The QR of calls that keep their arithmetic (set_kept_arithmetic): the grid form
// with a factorization in every pass, one column per step, a warp per row in the
// apply and a warp per entry in the sum of the shares. Its Q differs from the
// other forms' in the last bits only, and costs more (600 x 30 56 us against 48,
// 1600 x 50 97 and 78, 5760 x 90 314 and 265).

// 1/x for x in [1e-30, 1e30] (a pivot pre-scaled by an even power of two):
// an FP32 reciprocal seed (rcp.approx, relative error below 2^-22), then two
// Newton-Raphson steps r <- r + r (1 - x r) in FP64, each two fused
// multiply-adds (the error squares per step: 2^-22 -> 2^-44 -> FP64
// rounding). Two dependent FP64 instructions fewer than rsqrt_scaled, and its
// result is the multiplier 1/R_jj^2 the trailing update uses directly.
__device__ __forceinline__ double rcp_scaled(double x) {
  float f;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"((float)x));
  double r = (double)f;
  double e = fma(-x, r, 1.0);
  r = fma(r, e, r);
  e = fma(-x, r, 1.0);
  return fma(r, e, r);
}

// Warp reduction of the three convergence statistics; lane 0 holds the
// result. dev and dmax are maxima of non-negative doubles, taken on their bit
// patterns (integer order equals numeric order there), which keeps them off
// the FP64 unit.
__device__ __forceinline__ void warp_stats(long long &dev, long long &dmax, double &tr) {
  for (int o = 16; o > 0; o >>= 1) {
    dev = max(dev, __shfl_xor_sync(0xffffffffu, dev, o));
    dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
    tr += __shfl_xor_sync(0xffffffffu, tr, o);
  }
}

// Pivot step of column j (thread 0 only): R_jj = sqrt(pivot), stored as
// rinv2_j = 1/pivot, the multiplier of the trailing update, and the pivot
// itself; 1/R_jj is formed at publication, for all j at once and off the
// column chain. An exactly zero column of S (zero Gram diagonal) gets R_jj = 1,
// which leaves Q_j = 0 and couples nothing; sending it to the shifted attempt
// instead would make every pass shifted and leave ||Q^T Q - I|| at the shift
// (~1e-11) on an otherwise benign S. A pivot not safely positive fails the
// unshifted attempt; in the shifted attempt it sets the breakdown bit and is
// clamped so that nothing divides by zero.
// G is factorized scaled by sc = 2^-2k, which puts the largest Gram diagonal
// near 1 (exact: a power of two), so every pivot above the failure floor is a
// normal FP32 number and the chain carries no scaling; floor_piv and clamp
// (the value a failed pivot takes) are scaled alike.
__device__ __forceinline__ void chol_pivot(double *G, int ld, int j, const unsigned char *zero_col,
                                           double floor_piv, double clamp, int attempt,
                                           double *rinv2, double *pivots, unsigned char *fail,
                                           int *health) {
  if (zero_col[j]) {
    rinv2[j] = 1.0;
    pivots[j] = 1.0;
    return;
  }
  double piv = G[j * ld + j];
  if (!(piv > floor_piv)) {
    if (attempt == 0) fail[j] = 1;
    else atomicOr(health_word(health), kHealthBreakdown);
    piv = clamp;
  }
  pivots[j] = piv;
  rinv2[j] = (piv >= 1e-30 && piv <= 1e30) ? rcp_scaled(piv) : 1.0 / piv;
}

// Right-looking factorization with a one-column look-ahead: during the
// trailing update for column j, warp 0 first updates row j + 1 and thread 0
// takes the pivot of column j + 1 (the only serial step of the next column)
// while the other warps update the rest, so each column costs one barrier and
// the pivot's dependent FP64 chain overlaps the bulk of the update. Rows of R
// are not scaled in place: the update subtracts (G_ji y_j^2) G_jl, and the
// publication scales row j by y_j^2. G is read through L2 (__ldcg): in the
// fused form other blocks of the same launch wrote it.
__device__ __forceinline__ void chol_columns(const double *Gg, double *Ut_g, double *y_g, int c,
                                             int m, int *flags, double *sm, int *health) {
  const int ld = c + 1;
  double *G = sm;                                   // c x ld, upper triangle is updated
  __shared__ double s_red[3][kCholThreads / 32];
  __shared__ double s_diag_max, s_trace, s_dev, s_sc, s_unsc;
  __shared__ double s_rinv2[kMaxSmall];             // 1 / (sc R_jj^2)
  __shared__ double s_piv[kMaxSmall];               // sc R_jj^2 (the scaled pivot)
  __shared__ unsigned char s_zero[kMaxSmall];       // column j of S is exactly zero
  __shared__ unsigned char s_failc[kMaxSmall];      // unshifted pivot j not safely positive
  const int tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  const int tx = tid % 16, ty = tid / 16;           // 16 x 16 grid (kCholThreads = 256)

  // -- convergence test: G = I to working accuracy, except columns that are
  // exactly zero (a zero column stays zero through every pass). The test is
  // absolute on purpose: S of any scale (HaTT sketches of long chains reach
  // 1e-20 and below) is never mistaken for a converged basis.
  long long dev = 0, dmax = 0;          // bit patterns of non-negative doubles
  double tr = 0.0;
  int bad = 0;
  const int n = c * c;
  // entry e = i c + j of thread tid: (i, j) advanced by (di, dj) per step of
  // kCholThreads entries, with a carry, instead of a division per entry
  const int di = kCholThreads / c, dj = kCholThreads - (kCholThreads / c) * c;
  int ii = tid / c, jj = tid - (tid / c) * c;
  for (int e0 = tid; e0 < n; e0 += 4 * kCholThreads) {
    double v[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {         // four loads in flight per thread
      const int e = e0 + q * kCholThreads;
      v[q] = e < n ? __ldcg(Gg + e) : 0.0;
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int e = e0 + q * kCholThreads;
      if (e >= n) break;
      const int i = ii, j = jj;
      ii += di;
      jj += dj;
      if (jj >= c) {
        jj -= c;
        ++ii;
      }
      const long long bits = __double_as_longlong(fabs(v[q]));
      bad |= bits >= 0x7ff0000000000000LL;                   // Inf or NaN
      G[i * ld + j] = v[q];
      if (i == j) {
        s_zero[i] = (v[q] == 0.0);
        dmax = max(dmax, bits);
        tr += v[q];
        if (v[q] != 0.0) dev = max(dev, __double_as_longlong(fabs(v[q] - 1.0)));
      } else {
        dev = max(dev, bits);
      }
    }
  }
  warp_stats(dev, dmax, tr);
  if (lane == 0) {
    s_red[0][warp] = __longlong_as_double(dev);
    s_red[1][warp] = __longlong_as_double(dmax);
    s_red[2][warp] = tr;
  }
  // a non-finite Gram matrix (a non-finite input core or intermediate): record
  // it, leave S as it is and stop this QR (every later pass is a no-op)
  if (__syncthreads_or(bad)) {
    if (tid == 0) {
      atomicOr(health_word(health), kHealthNonfinite);
      flags[0] = 1;
      flags[1] = 1;
    }
    return;
  }
  if (tid == 0) {
    double d0 = 0.0, d1 = 0.0, d2 = 0.0;
    for (int w = 0; w < kCholThreads / 32; ++w) {
      d0 = fmax(d0, s_red[0][w]);
      d1 = fmax(d1, s_red[1][w]);
      d2 += s_red[2][w];
    }
    s_dev = d0;
    s_diag_max = d1;
    s_trace = d2;
    // pivot scaling 2^-2k with the largest diagonal in [0.5, 2) after scaling;
    // the exponent is read off the bits (frexp / ldexp are long sequences on
    // this chain), with frexp / ldexp kept for subnormal or extreme values
    const long long bits = __double_as_longlong(d1);
    const int be = (int)((bits >> 52) & 0x7ff);
    int ex = 0;
    if (be > 0) ex = be - 1022;                 // d1 = m 2^ex, m in [0.5, 1)
    else if (d1 > 0.0) frexp(d1, &ex);
    const int k = ex / 2;
    s_sc = (-2 * k + 1023 >= 1 && -2 * k + 1023 <= 2046)
               ? __longlong_as_double((long long)(-2 * k + 1023) << 52) : ldexp(1.0, -2 * k);
    s_unsc = (-k + 1023 >= 1 && -k + 1023 <= 2046)
                 ? __longlong_as_double((long long)(-k + 1023) << 52) : ldexp(1.0, -k);
  }
  __syncthreads();
  const double u = 1.1102230246251565e-16;
  const double sc = s_sc, unsc = s_unsc;
  if (s_dev <= 8.0 * c * u) {              // already orthonormal: nothing to apply
    if (tid == 0) { flags[0] = 1; flags[1] = 1; }
    return;
  }
  for (int i = ty; i < c; i += 16)         // the factorization runs on sc G
    for (int j = tx; j < c; j += 16) G[i * ld + j] *= sc;

  // -- Cholesky: first unshifted, then shifted if a pivot is not safely positive.
  // A failed pivot of column j is recorded in s_failc[j] while column j - 1
  // is updated and read by every thread after that column's barrier, so all
  // threads leave the column loop at the same j.
  for (int attempt = 0; attempt < 2; ++attempt) {
    double shift = 0.0;
    if (attempt == 1) {
      shift = 11.0 * ((double)m * c + (double)c * (c + 1)) * u * s_trace;
      if (!(shift > 0.0)) shift = 1e-300;
      for (int e = tid; e < c * c; e += kCholThreads) {
        const int i = e / c, j = e % c;
        G[i * ld + j] = (__ldcg(Gg + e) + (i == j ? shift : 0.0)) * sc;
      }
      if (tid == 0) flags[3] += 1;
    }
    for (int j = tid; j < c; j += kCholThreads) s_failc[j] = 0;
    __syncthreads();
    const double floor_piv = (attempt == 0) ? (double)c * u * s_diag_max * sc : 0.0;
    const double clamp = fmax(shift, 1e-300) * sc;
    if (tid == 0) chol_pivot(G, ld, 0, s_zero, floor_piv, clamp, attempt, s_rinv2, s_piv, s_failc, health);
    __syncthreads();
    bool failed = false;
    for (int j = 0; j < c; ++j) {
      if (s_failc[j]) {
        failed = true;
        break;
      }
      const double y2 = s_rinv2[j];
      const double *rowj = G + j * ld;
      if (warp == 0 && j + 1 < c) {       // look-ahead: row j + 1, then its pivot
        const int i = j + 1;
        const double rji = rowj[i] * y2;
        for (int l = i + lane; l < c; l += 32) G[i * ld + l] = fma(-rji, rowj[l], G[i * ld + l]);
        __syncwarp();
        if (lane == 0) chol_pivot(G, ld, i, s_zero, floor_piv, clamp, attempt, s_rinv2, s_piv, s_failc, health);
      }
      // trailing update of the rows below by warps 1..7 on a 14 x 16 grid:
      // warp 0 carries the pivot chain and takes no share of it
      if (warp > 0) {
        const int bt = tid - 32, bx = bt % 16, by = bt / 16;
        for (int i = j + 2 + by; i < c; i += 14) {
          const double rji = rowj[i] * y2;
          for (int l = i + bx; l < c; l += 16) G[i * ld + l] = fma(-rji, rowj[l], G[i * ld + l]);
        }
      }
      __syncthreads();
    }
    if (!failed) break;
    __syncthreads();                      // all reads of G and s_failc done before the retry
  }

  // -- publish R = D U~ as the unit upper triangle U~ (U~_jl = R_jl / R_jj =
  // G_jl / G_jj with G the updated, scaled Gram row: the scale cancels) and
  // y_j = 1 / R_jj; the apply
  // kernel solves with them, so no serial triangular inverse is formed in
  // this single block
  for (int i = ty; i < c; i += 16) {
    const double yi2 = s_rinv2[i];
    for (int l = tx; l < c; l += 16)
      Ut_g[i * c + l] = (l > i) ? G[i * ld + l] * yi2 : (l == i ? 1.0 : 0.0);
  }
  for (int i = tid; i < c; i += kCholThreads) {
    double yi = 1.0;                      // 1 / R_ii (1 for an exactly zero column)
    if (!s_zero[i]) {                     // the pivot is sc R_ii^2, sc = unsc^2
      const double ps = s_piv[i];
      yi = ((ps >= 1e-30 && ps <= 1e30) ? rsqrt_scaled(ps) : rsqrt_newton(ps)) * unsc;
    }
    y_g[i] = yi;
  }
  // this pass applies; ||G - I||_max <= 0.1/c puts every eigenvalue of G in
  // [0.9, 1.1] (Gerschgorin): one more Cholesky QR pass orthonormalizes to
  // working accuracy, so this pass is the last one. Written last: the
  // read-modify-write would otherwise sit on the first pivot's path.
  if (tid == 0) {
    flags[1] = 0;
    flags[2] += 1;
    if (s_dev <= 0.1 / c) flags[0] = 1;
  }
}

// Two rows at once, their chains interleaved (the same operations on each
// row as trsm_row, so a row's result does not depend on its partner).
template <int NS>
__device__ __forceinline__ void trsm_row2(double (&x)[4], double (&z)[4], const double *Us, int c,
                                          int lane) {
#pragma unroll
  for (int s0 = 0; s0 < NS; ++s0) {
    const int lend = min(c, 32 * (s0 + 1));
    for (int l = 32 * s0; l < lend; ++l) {
      const double xl = __shfl_sync(0xffffffffu, x[s0], l & 31);
      const double zl = __shfl_sync(0xffffffffu, z[s0], l & 31);
      const double *u = Us + l * c;
#pragma unroll
      for (int s = s0; s < NS; ++s) {
        const int col = lane + 32 * s;
        if (col > l && col < c) {
          const double uv = u[col];
          x[s] = fma(-xl, uv, x[s]);
          z[s] = fma(-zl, uv, z[s]);
        }
      }
    }
  }
}

__device__ __forceinline__ void apply_warp_rows(double *S, long long ldS, int c, const double *Us,
                                                const double *ys, int r_first, int r_end, int r_step) {
  const int lane = threadIdx.x & 31;
  const int ns = (c + 31) / 32;          // column slots in use (c <= 128)
  for (int r = r_first; r < r_end; r += 2 * r_step) {
    double *row = S + (long long)r * ldS;
    double *row2 = S + (long long)(r + r_step) * ldS;
    const bool two = r + r_step < r_end;   // the warp's next row: solved alongside
    double x[4], z[4];
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const bool in = s < ns && lane + 32 * s < c;
      x[s] = in ? row[lane + 32 * s] : 0.0;
      z[s] = (in && two) ? row2[lane + 32 * s] : 0.0;
    }
    if (two) {
      switch (ns) {
        case 1: trsm_row2<1>(x, z, Us, c, lane); break;
        case 2: trsm_row2<2>(x, z, Us, c, lane); break;
        case 3: trsm_row2<3>(x, z, Us, c, lane); break;
        default: trsm_row2<4>(x, z, Us, c, lane); break;
      }
    } else {
      switch (ns) {
        case 1: trsm_row<1>(x, Us, c, lane); break;
        case 2: trsm_row<2>(x, Us, c, lane); break;
        case 3: trsm_row<3>(x, Us, c, lane); break;
        default: trsm_row<4>(x, Us, c, lane); break;
      }
    }
#pragma unroll
    for (int s = 0; s < 4; ++s) {
      const int col = lane + 32 * s;
      if (s < ns && col < c) {
        row[col] = x[s] * ys[col];
        if (two) row2[col] = z[s] * ys[col];
      }
    }
  }
}

// Entry t of G summed over the nb shares by one warp: lanes over shares in
// order, then a fixed shuffle tree; lane 0 writes G(i, j) and G(j, i).
__device__ __forceinline__ void gram_entry(const double *part, int nb, int c, int t, double *G) {
  const int lane = threadIdx.x & 31;
  const int T = c * (c + 1) / 2;
  constexpr int kPer = (kQrMaxBlocks + 31) / 32;
  double sh[kPer];                        // all loads in flight, then summed in share order
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    const int p = lane + 32 * k;
    sh[k] = p < nb ? __ldcg(part + (long long)p * T + t) : 0.0;
  }
  double v = 0.0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) v += sh[k];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) {
    int i, j;
    upper_index(t, c, i, j);
    G[i * c + j] = v;
    G[j * c + i] = v;
  }
}

template <int MAXQ>
__global__ void __launch_bounds__(kCholThreads, 1)
qr_columns_kernel(double *S, int m, int c, long long ldS, double *G, double *Ut, double *y,
                  double *part, int *flags, int *health, long long spin_cap) {
  pdl_enter();
  extern __shared__ double sm[];
  const int tid = threadIdx.x, warp = tid >> 5;
  constexpr int kWarps = kCholThreads / 32;
  const int nb = gridDim.x, bid = blockIdx.x;
  const int per = (m + nb - 1) / nb;
  const int r0 = min(m, bid * per), r1 = min(m, r0 + per);
  const int T = c * (c + 1) / 2;
  GramSlots<MAXQ> g;
  gram_slots(c, g);
  int *bar = flags + 4;
  int epoch = 0;
  for (int pass = 0; pass < kPasses; ++pass) {
    gram_share(S, ldS, c, r0, r1, g, part + (long long)bid * T, sm);
    if (!grid_barrier(bar, epoch, spin_cap)) return;
    for (int t = bid * kWarps + warp; t < T; t += nb * kWarps) gram_entry(part, nb, c, t, G);
    if (!grid_barrier(bar, epoch, spin_cap)) return;
    if (bid == 0) chol_columns(G, Ut, y, c, m, flags, sm, health);
    if (!grid_barrier(bar, epoch, spin_cap)) return;
    const int done = __ldcg(flags), skip = __ldcg(flags + 1);
    if (skip) return;                      // orthonormal already (or a non-finite G)
    for (int e = tid; e < c * c; e += kCholThreads) sm[e] = __ldcg(Ut + e);
    for (int e = tid; e < c; e += kCholThreads) sm[c * c + e] = __ldcg(y + e);
    __syncthreads();
    apply_warp_rows(S, ldS, c, sm, sm + c * c, r0 + warp, r1, kWarps);
    if (done) return;                      // this pass was the last one
    if (!grid_barrier(bar, epoch, spin_cap)) return;
  }
}

// SMs and cooperative-launch support of the current device, cached per
// device (0 SMs: unknown device).
void device_info(int &sms, bool &coop) {
  static int s_sms[64] = {};
  static signed char s_coop[64] = {};
  sms = 0;
  coop = false;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    return;
  }
  if (s_sms[dev] == 0) {
    int n = 0, co = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&co, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      return;
    }
    s_coop[dev] = co ? 1 : 0;
    s_sms[dev] = n;
  }
  sms = s_sms[dev];
  coop = s_coop[dev] != 0;
}

// Sizes for the cluster form: up to m c^2 / 2 = 32 k multiply-adds. Measured (us,
// cluster and grid): 96 x 12 26 and 38, 160 x 20 37.5 and ~37, 400 x 20 49 and
// 38.5, 256 x 32 60 and 48.
bool cluster_sized(int m, int c) { return (long long)m * (c * (c + 1) / 2) <= kClusterFma; }

// Blocks (Gram shares) of a QR of m rows: at least kQrMinRows rows each, at
// most one per SM (the grid form keeps every block resident).
int grid_blocks(int m, int sms) {
  const int want = (m + kQrMinRows - 1) / kQrMinRows;
  return std::max(1, std::min({want, std::max(sms, 1), kQrMaxBlocks}));
}
int qr_blocks(int m, int c, int sms) {
  if (!cluster_sized(m, c)) return grid_blocks(m, sms);
  const int want = (m + kQrMinRows - 1) / kQrMinRows;
  int nb = kClusterBlocks;
  while (nb / 2 >= want) nb /= 2;
  return nb;
}

// Test hooks, read once: HATT_QR_FORM=steps makes single calls use the
// launch-per-step form; HATT_QR_SPIN_CAP=<n> bounds each grid-barrier wait of
// the fused form to n polls (a small n makes the waits run out: the timeout
// status without a hang).
bool force_qr_steps() {
  static const bool v = [] {
    const char *e = getenv("HATT_QR_FORM");
    return e != nullptr && strcmp(e, "steps") == 0;
  }();
  return v;
}

long long qr_spin_cap() {
  static const long long v = [] {
    const char *e = getenv("HATT_QR_SPIN_CAP");
    const long long n = e ? atoll(e) : 0;
    return n > 0 ? n : kQrSpinCap;
  }();
  return v;
}

size_t chol_smem(int c) { return (size_t)c * (c + 1) * sizeof(double); }
size_t trsm_smem(int c) { return (size_t)(c * c + c) * sizeof(double); }
size_t gram_smem(int c) { return (size_t)kQrRowTile * c * sizeof(double); }
size_t fused_smem(int c) { return std::max((size_t)c * (c + 2) * sizeof(double), gram_smem(c)); }

QrTol qr_tol(int c) {
  const double u = 1.1102230246251565e-16;
  const double t[3] = {8.0 * c * u, std::sqrt(u / c), 0.1 / c};
  QrTol r;
  memcpy(&r.orth, &t[0], sizeof(double));
  memcpy(&r.linear, &t[1], sizeof(double));
  memcpy(&r.last, &t[2], sizeof(double));
  return r;
}

}  // namespace

cudaError_t qr_health_word(int *value, bool clear) {
  cudaError_t e = cudaMemcpyFromSymbol(value, g_qr_health, sizeof(int));
  if (e == cudaSuccess && clear && *value != 0) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(g_qr_health, &zero, sizeof(int));
  }
  return e;
}

// G, U~, y, then the blocks' Gram shares.
size_t qr_scratch_doubles(int m, int c) {
  (void)m;
  return (size_t)2 * c * c + c + (size_t)kQrMaxBlocks * c * (c + 1) / 2;
}

cudaError_t qr_inplace(double *S, int m, int c, long long ldS, double *scratch, int *flags,
                       cudaStream_t st) {
  if (c <= 0 || m <= 0) return cudaSuccess;
  if (c > kMaxSmall) return cudaErrorInvalidValue;
  double *G = scratch;
  double *Ut = scratch + (size_t)c * c;
  double *y = scratch + (size_t)2 * c * c;
  double *part = scratch + (size_t)2 * c * c + c;
  int sms = 0;
  bool coop = false;
  device_info(sms, coop);
  if (sms <= 0) return cudaErrorInvalidDevice;
  const int nb = qr_blocks(m, c, sms);
  const QrTol tol = qr_tol(c);
  const bool small = c <= 64;               // the kQrSlots64 instantiations
  const bool cluster = cluster_sized(m, c) && qr_spin_cap() == kQrSpinCap;
  cudaError_t e = cudaSuccess;
  if (kept_arithmetic() && coop && programmatic_launch() && !force_qr_steps()) {
    auto kernel = small ? qr_columns_kernel<kQrSlots64> : qr_columns_kernel<kQrMaxSlots>;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused_smem(kMaxSmall));
    if (e == cudaSuccess) e = cudaMemsetAsync(flags, 0, 6 * sizeof(int), st);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.numAttrs = 1;
    cfg.gridDim = dim3(grid_blocks(m, sms));
    cfg.blockDim = dim3(kCholThreads);
    cfg.dynamicSmemBytes = fused_smem(c);
    cfg.stream = st;
    cfg.attrs = attr;
    e = cudaLaunchKernelEx(&cfg, kernel, S, m, c, ldS, G, Ut, y, part, flags, health_target(), qr_spin_cap());
    note_launch();
    return e;
  }
  if (!force_qr_steps() && (cluster || (coop && programmatic_launch()))) {
    auto kernel = cluster ? (small ? qr_fused_kernel<kQrSlots64, true> : qr_fused_kernel<kQrMaxSlots, true>)
                          : (small ? qr_fused_kernel<kQrSlots64, false> : qr_fused_kernel<kQrMaxSlots, false>);
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fused_smem(kMaxSmall));
    if (e == cudaSuccess && !cluster) e = cudaMemsetAsync(flags, 0, 6 * sizeof(int), st);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr[2];
    cudaLaunchConfig_t cfg = {};
    if (cluster) {
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = nb;
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      attr[1].val.programmaticStreamSerializationAllowed = 1;
      cfg.numAttrs = programmatic_launch() ? 2 : 1;
    } else {
      attr[0].id = cudaLaunchAttributeCooperative;
      attr[0].val.cooperative = 1;
      cfg.numAttrs = 1;
    }
    cfg.gridDim = dim3(nb);
    cfg.blockDim = dim3(kCholThreads);
    cfg.dynamicSmemBytes = fused_smem(c);
    cfg.stream = st;
    cfg.attrs = attr;
    e = cudaLaunchKernelEx(&cfg, kernel, S, m, c, ldS, G, Ut, y, part, tol, flags, health_target(),
                           qr_spin_cap());
    note_launch();
    return e;
  }
  e = cudaMemsetAsync(flags, 0, 6 * sizeof(int), st);
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(chol_inv_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)chol_smem(kMaxSmall));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(trsm_rows_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)trsm_smem(kMaxSmall));
  if (e != cudaSuccess) return e;
  const int T = c * (c + 1) / 2;
  const int sum_blocks = std::max(1, std::min((T + 7) / 8, 2 * sms));
  const int blocks = std::max(1, std::min((m + kTrsmThreads / 32 - 1) / (kTrsmThreads / 32), 2 * sms));
  for (int p = 0; p < kPasses; ++p) {
    launch_k(small ? gram_share_kernel<kQrSlots64> : gram_share_kernel<kQrMaxSlots>, nb,
             kCholThreads, gram_smem(c), st, S, ldS, m, c, part, flags);
    note_launch();
    launch_k(gram_sum_kernel, sum_blocks, kCholThreads, 0, st, part, nb, c, G, flags);
    note_launch();
    launch_k(chol_inv_kernel, 1, kCholThreads, chol_smem(c), st, G, Ut, y, c, m, tol, flags, health_target());
    note_launch();
    launch_k(trsm_rows_kernel, blocks, kTrsmThreads, trsm_smem(c), st, S, m, c, ldS, Ut, y, flags);
    note_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace hatt
