// FP32 start of the symmetric eigen solver where no tolerance is set:
// eigenvectors of a c x c matrix (c <= 128) in one block, the seed of the FP64
// refinement (k_refine.cu).
//
//   1. Householder tridiagonalization (Golub & Van Loan 8.3.1) with the whole
//      matrix in registers: warp w holds rows w, w + 16, ..., lane l columns
//      l, l + 32, ...; row k of the symmetric trailing block is the column the
//      next reflector needs, so its warp forms it by shuffles. Two barriers per
//      column: after the reflector, and after p = beta A v (the dot products of
//      a warp's rows are reduced together: 9 shuffles for 8 rows, not 40).
//   2. eigenvalues by multisection on Sturm counts, a group of lanes per
//      eigenvalue;
//   3. eigenvectors of the tridiagonal matrix by two steps of inverse iteration,
//      one thread per vector: the elimination with partial pivoting (Golub & Van
//      Loan 4.3) is done once and its multipliers are kept for the second step;
//   4. modified Gram-Schmidt inside clusters of eigenvalues closer than 1e-3 of
//      the spectral radius, where inverse iteration alone does not give
//      orthogonal vectors: vectors in registers (warp w: w, w + 16, ...), one
//      barrier per finished vector; a second sweep where a vector lost more than
//      half of its squared length;
//   5. back-transformation by the stored reflectors, four lanes per column.
// Columns come out sorted by decreasing eigenvalue. The result only seeds the
// refinement, which needs a relative residual of ~1e-5 and an orthogonal start.
//
// Measured (clocks at c = 50, random spectrum; eig_tridiag32_kernel of k_trunc.cu
// in parentheses): tridiagonalization 56 k (112 k), eigenvalues 15 k (38 k),
// inverse iteration 23 k (30 k), back-transformation 14 k (24 k), 58 us in all
// (116); c = 90: 124 us (400), a graded spectrum's Gram-Schmidt 85 us of 209.
//
// Bound: dependent chains of one block (barriers, shuffles, reciprocals), not
// arithmetic: 16 warps, so that no chain waits for another's issue slots, and
// no FP64 instruction (a warp-wide one holds the SM's FP64 unit for 16 clocks):
// conversions work on the bits.
#include <algorithm>
#include <type_traits>
#include "hatt_internal.cuh"

namespace hatt {
namespace {

constexpr int kT = 512;
constexpr int kW = kT / 32;
constexpr float kClusterRel = 1e-3f;
constexpr int kBatch = 32;               // vectors per inverse-iteration batch where c > 96

template <int CT>
__host__ __device__ constexpr int inv_batch() { return CT == 4 ? kBatch : 32 * CT; }

// Shared memory (floats): reflectors c x 32 CT, eigenvectors c x (c | 1), and
// the four factor arrays of an inverse-iteration batch, c x (batch | 1) each.
template <int CT>
size_t eig_smem(int c) {
  const int nb = std::min(c, inv_batch<CT>());
  return ((size_t)c * 32 * CT + (size_t)c * (c | 1) + (size_t)4 * c * (nb | 1)) * sizeof(float);
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Sums of R (4 or 8) values over the warp: on return every lane holds the sum
// of value index_of_lane<R>(lane).
template <int R>
__device__ __forceinline__ float warp_sums(const float (&v)[R], int lane) {
  float x[R];
#pragma unroll
  for (int i = 0; i < R; ++i) x[i] = v[i];
  int n = R, o = 16;
#pragma unroll
  for (int lev = 0; lev < (R == 8 ? 3 : 2); ++lev) {
    const bool up = (lane & o) != 0;
    n >>= 1;
#pragma unroll
    for (int i = 0; i < R / 2; ++i)
      if (i < n) {
        const float keep = up ? x[i + n] : x[i], send = up ? x[i] : x[i + n];
        x[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    o >>= 1;
  }
  float s = x[0];
  for (; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}
template <int R>
__device__ __forceinline__ int index_of_lane(int lane) {
  return R == 8 ? ((lane >> 4) & 1) * 4 + ((lane >> 3) & 1) * 2 + ((lane >> 2) & 1)
                : ((lane >> 4) & 1) * 2 + ((lane >> 3) & 1);
}
template <int R>
__device__ __forceinline__ bool leads_index(int lane) { return (lane & (R == 8 ? 3 : 7)) == 0; }

// x 2^-s rounded to FP32 on the bits; below the FP32 normal range 0, above it
// (and for an infinity or NaN) the largest exponent.
__device__ __forceinline__ float to_f32(double x, int s) {
  const unsigned long long b = ((unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull) + (1ull << 28);
  const int e = (int)(b >> 52) - 896 - s;
  const unsigned m = (unsigned)(b >> 29) & 0x7FFFFFu;
  const unsigned sign = (unsigned)__double2hiint(x) & 0x80000000u;
  return e <= 0 ? 0.0f : __uint_as_float(sign | ((unsigned)min(e, 254) << 23) | m);
}
// FP32 to FP64 on the bits (zero and subnormal give zero).
__device__ __forceinline__ double to_f64(float x) {
  const unsigned u = __float_as_uint(x), e = (u >> 23) & 0xFFu;
  if (e == 0) return 0.0;
  const unsigned hi = (u & 0x80000000u) | ((e + 896u) << 20) | ((u >> 3) & 0xFFFFFu);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// Entry j of the start vector of eigenvector i: a hash of (i, j) mapped to
// [-1, 1). Start vectors must have independent projections on a cluster's
// eigenspace; a smooth pattern close to the all-ones vector does not (all of
// them project onto nearly the same direction), and Gram-Schmidt then keeps
// mostly the out-of-cluster error.
__device__ __forceinline__ float start_entry(int i, int j) {
  unsigned h = (unsigned)i * 0x9E3779B1u + (unsigned)j * 0x85EBCA77u + 0x165667B1u;
  h ^= h >> 15;
  h *= 0x2C1B3C6Du;
  h ^= h >> 12;
  h *= 0x297A2D39u;
  h ^= h >> 15;
  return -1.0f + 2.0f * (float)(h & 0xffffffu) * (1.0f / 16777216.0f);
}

// Back substitution of the factored shifted matrix (rp: reciprocal pivots, du,
// du2: the two upper diagonals), z in place, one vector with stride ld; the next
// row's loads are issued before this row's store.
// Whenever a component exceeds 1e18 the whole vector (solved and pending parts)
// is scaled by 1e-18: the system is linear, only the direction of z matters, and
// a shift equal to an eigenvalue leaves a pivot near zero.
__device__ __forceinline__ void back_solve(float *z, int ldz, const float *rp, const float *du,
                                           const float *du2, int ld, int c) {
  float z1 = 0.0f, z2 = 0.0f;
  int j = c - 1;
  float r = rp[j * ld], u = du[j * ld], u2 = du2[j * ld], b = z[j * ldz];
  for (; j >= 0; --j) {
    const int jn = max(j - 1, 0);
    const float rn = rp[jn * ld], un = du[jn * ld], u2n = du2[jn * ld];
    float bn = z[jn * ldz];
    float t = fmaf(-u, z1, fmaf(-u2, z2, b)) * r;
    if (fabsf(t) > 1e18f) {
      for (int q = 0; q < c; ++q) z[q * ldz] *= 1e-18f;
      bn *= 1e-18f;
      z1 *= 1e-18f;
      t *= 1e-18f;
    }
    z[j * ldz] = t;
    z2 = z1;
    z1 = t;
    r = rn;
    u = un;
    u2 = u2n;
    b = bn;
  }
}

template <int CT>
__global__ void __launch_bounds__(kT, 1)
eig_start_kernel(const double *G, int c, double *U, const int *skip) {
  pdl_enter();
  if (skip && *skip) return;
  constexpr int R = CT <= 2 ? 4 : 8;     // rows per warp, padded to a power of two
  constexpr int LDV = 32 * CT;
  extern __shared__ __align__(16) float fs[];
  float *Vh = fs;                        // reflector k in row k, zero up to entry k
  float *Z = Vh + c * LDV;               // c x ldz, eigenvectors (columns)
  const int ldz = c | 1;
  float *fac = Z + c * ldz;              // inverse iteration
  __shared__ float d[130], e[130], tau[128], lam[128], p[128];   // d, e: two zeros past the end
  __shared__ float2 de[128];             // (d_j, e_{j-1}^2)
  __shared__ float s_zb[2][128];         // a finished vector of the Gram-Schmidt sweep, two buffers
  __shared__ float s_lo, s_hi;
  __shared__ int s_cnt[kT];
  __shared__ int s_emax, s_again, s_end[129], s_list[128], s_count;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // the matrix, scaled by a power of two so that its largest diagonal is in [1/2, 1)
  if (tid == 0) s_emax = 0;
  if (tid < 128) p[tid] = 0.0f;
  __syncthreads();
  if (tid < c) atomicMax(&s_emax, (__double2hiint(G[tid * c + tid]) >> 20) & 0x7ff);
  __syncthreads();
  const int sc = s_emax - 1022;
  float a[R][CT];
#pragma unroll
  for (int q = 0; q < R; ++q)
#pragma unroll
    for (int t = 0; t < CT; ++t) {
      const int i = warp + kW * q, j = lane + 32 * t;
      a[q][t] = (i < c && j < c) ? to_f32(G[i * c + j], sc) : 0.0f;
    }

  // 1. tridiagonalization, column k = 16 qb + kk: the row a warp holds for it is
  // its qb-th, a compile-time register index (a selection among all of a warp's
  // rows cost 1000 to 2900 clocks per column). Finished rows drop out; finished
  // columns keep being transformed (by reflectors that vanish there: they stay
  // bounded) and are never read again.
  auto columns = [&](auto block) {
    constexpr int qb = decltype(block)::value;
#pragma unroll 1
    for (int kk = 0; kk < kW; ++kk) {
      const int k = kW * qb + kk;
      if (k + 2 >= c) break;
      if (warp == kk) {                  // reflector of column k, from row k
        float x[CT], s2 = 0.0f, x0 = 0.0f, dk = 0.0f;
#pragma unroll
        for (int t = 0; t < CT; ++t) {
          const int j = lane + 32 * t;
          x[t] = a[qb][t];
          if (t == (k + 1) >> 5) x0 = x[t];
          if (t == k >> 5) dk = x[t];
          x[t] = j > k ? x[t] : 0.0f;
          s2 = fmaf(x[t], x[t], s2);
        }
        x0 = __shfl_sync(0xffffffffu, x0, (k + 1) & 31);
        s2 = warp_sum(s2);
        const bool none = !(s2 > 1e-36f);
        const float alpha = none ? x0 : -copysignf(s2 * rsqrtf(s2), x0);
        const float v0 = x0 - alpha;
        const float vtv = s2 - x0 * x0 + v0 * v0;
#pragma unroll
        for (int t = 0; t < CT; ++t) {
          const int j = lane + 32 * t;
          Vh[k * LDV + j] = none ? 0.0f : (j == k + 1 ? v0 : x[t]);
        }
        if (lane == (k & 31)) d[k] = dk;
        if (lane == 0) {
          e[k] = alpha;
          tau[k] = (none || !(vtv > 0.0f)) ? 0.0f : __fdividef(2.0f, vtv);
        }
      }
      __syncthreads();
      const float beta = tau[k];
      float v[CT], acc[R];
#pragma unroll
      for (int t = 0; t < CT; ++t) v[t] = Vh[k * LDV + lane + 32 * t];
#pragma unroll
      for (int q = 0; q < R; ++q) {
        acc[q] = 0.0f;
        if (q >= qb && kW * q < LDV) {
#pragma unroll
          for (int t = 0; t < CT; ++t) acc[q] = fmaf(a[q][t], v[t], acc[q]);
        }
      }
      const float ps = warp_sums<R>(acc, lane);
      if (leads_index<R>(lane)) {
        const int i = warp + kW * index_of_lane<R>(lane);
        if (i < 128) p[i] = beta * ps;
      }
      __syncthreads();
      float w[CT], kd = 0.0f;
#pragma unroll
      for (int t = 0; t < CT; ++t) {
        w[t] = p[lane + 32 * t];
        kd = fmaf(v[t], w[t], kd);
      }
      const float K = 0.5f * beta * warp_sum(kd);
#pragma unroll
      for (int t = 0; t < CT; ++t) w[t] = fmaf(-K, v[t], w[t]);
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (q >= qb && kW * q < LDV) {
          const int i = warp + kW * q;
          const float vi = Vh[k * LDV + i], wi = fmaf(-K, vi, p[i]);
#pragma unroll
          for (int t = 0; t < CT; ++t) a[q][t] = fmaf(-wi, v[t], fmaf(-vi, w[t], a[q][t]));
        }
    }
  };
  columns(std::integral_constant<int, 0>{});
  columns(std::integral_constant<int, 1>{});
  columns(std::integral_constant<int, 2>{});
  columns(std::integral_constant<int, 3>{});
  if constexpr (R == 8) {
    columns(std::integral_constant<int, 4>{});
    columns(std::integral_constant<int, 5>{});
    columns(std::integral_constant<int, 6>{});
    columns(std::integral_constant<int, 7>{});
  }
#pragma unroll
  for (int q = 0; q < R; ++q)
#pragma unroll
    for (int t = 0; t < CT; ++t) {
      const int i = warp + kW * q, j = lane + 32 * t;
      if (i < c && i >= c - 2 && j == i) d[i] = a[q][t];
      if (c >= 2 && i == c - 1 && j == c - 2) e[c - 2] = a[q][t];
    }
  if (tid == 0) {
    e[c - 1] = e[c] = e[c + 1] = 0.0f;
    d[c] = d[c + 1] = 0.0f;
    s_again = 0;
    s_count = 0;
  }
  __syncthreads();

  // Gerschgorin interval (warp 0). e^2 is kept away from zero, so that the
  // Sturm recurrence below never forms 0 * infinity
  if (tid < c) de[tid] = make_float2(d[tid], tid > 0 ? fmaxf(e[tid - 1] * e[tid - 1], 1e-36f) : 0.0f);
  if (warp == 0) {
    float lo = 3.0e38f, hi = -3.0e38f;
    for (int i = lane; i < c; i += 32) {
      const float r = (i > 0 ? fabsf(e[i - 1]) : 0.0f) + fabsf(e[i]);
      lo = fminf(lo, d[i] - r);
      hi = fmaxf(hi, d[i] + r);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if (lane == 0) {
      s_lo = lo;
      s_hi = hi;
    }
  }
  __syncthreads();

  // 2. eigenvalues. The number of eigenvalues below x is the number of negative
  // pivots q_j = d_j - x - e_{j-1}^2 / q_{j-1}; a zero pivot gives an infinite and
  // then a regular one. First every thread counts at its own point of the
  // interval, which brackets all eigenvalues 512 times closer; then a group of g
  // lanes per eigenvalue shrinks its bracket g + 1 times per round (bound: the
  // reciprocal unit, 16 lanes per clock, and its latency).
  const float glo = s_lo, ghi = s_hi;
  const float span = fmaxf(fabsf(glo), fabsf(ghi));
  auto count_below = [&](float x) {
    float q = de[0].x - x;
    int n = q < 0.0f;
#pragma unroll 4
    for (int j = 1; j < c; ++j) {
      const float2 f = de[j];
      float r;
      asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(q));
      q = fmaf(-f.y, r, f.x - x);
      n += (int)(__float_as_uint(q) >> 31);
    }
    return n;
  };
  {
    constexpr float step = 1.0f / (float)(kT + 1);
    s_cnt[tid] = count_below(fmaf(ghi - glo, (float)(tid + 1) * step, glo));
    __syncthreads();
    constexpr int g = CT <= 2 ? 8 : 4;   // lanes per eigenvalue
    const int i = tid / g, l = tid % g;
    const int target = c - 1 - i;        // count of smaller eigenvalues
    int below = 0;                       // points whose count is at most the target
    for (int s = kT / 2; s > 0; s >>= 1)
      if (s_cnt[below + s - 1] <= target) below += s;
    if (below == kT - 1 && s_cnt[kT - 1] <= target) below = kT;
    float x0 = below == 0 ? glo : fmaf(ghi - glo, (float)below * step, glo);
    float x1 = below == kT ? ghi : fmaf(ghi - glo, (float)(below + 1) * step, glo);
    bool active = i < c;
    constexpr float inv_n = 1.0f / (float)(g + 1);
#pragma unroll 1
    for (int round = 0; round < 64 && __any_sync(0xffffffffu, active); ++round) {
      const float x = fmaf(x1 - x0, (float)(l + 1) * inv_n, x0);
      float na = x0, nb = x1;
      if (count_below(x) <= target) na = x;
      else nb = x;
#pragma unroll
      for (int o = 1; o < g; o <<= 1) {
        na = fmaxf(na, __shfl_xor_sync(0xffffffffu, na, o));
        nb = fminf(nb, __shfl_xor_sync(0xffffffffu, nb, o));
      }
      if (active) {
        x0 = na;
        x1 = nb;
        // the tridiagonal matrix itself is known to ~1e-7 of its span
        if (x1 - x0 <= 2.4e-7f * fmaxf(fmaxf(fabsf(x0), fabsf(x1)), 1e-4f * span)) active = false;
      }
    }
    if (i < c && l == 0) lam[i] = 0.5f * (x0 + x1);
  }
  __syncthreads();
  // Shifts of equal (or nearly equal) eigenvalues are moved apart by 10 ulps
  // of the larger magnitude, as in LAPACK's inverse iteration: identical
  // shifts meet the same near-zero pivot and return the same vector, which
  // Gram-Schmidt would then annihilate (exact ties occur, e.g. the two equal
  // singular values of sin(a + b) = sin a cos b + cos a sin b).
  if (tid == 0) {
    float prev = lam[0];
    for (int i = 1; i < c; ++i) {
      const float pert = 6e-7f * fabsf(prev);
      float x = lam[i];
      if (prev - x < pert) {
        x = prev - pert;
        lam[i] = x;
      }
      prev = x;
    }
  }
  __syncthreads();

  // 3. inverse iteration, one thread per eigenvector (column i of Z). Factors
  // and right-hand sides lie [row][vector]: lanes are neighbouring vectors.
  const float tiny = 1e-30f + 1e-13f * span;
  const int nb = min(c, inv_batch<CT>()), ldf = nb | 1;
  for (int j = warp; j < c; j += kW)
    for (int i = lane; i < c; i += 32) Z[j * ldz + i] = start_entry(i, j);
  __syncthreads();
#pragma unroll 1
  for (int i0 = 0; i0 < c; i0 += nb) {
    const int il = tid, i = i0 + il;
    const bool on = il < nb && i < c;
    float *rp = fac + il, *du = rp + c * ldf, *du2 = du + c * ldf, *fm = du2 + c * ldf;
    float *z = Z + i;
    if (on) {
      // elimination of T - lam I; the pivoting choice is made with selects, the
      // lanes solve different systems. The low bit of a multiplier says that the
      // rows were not swapped.
      const float l = lam[i];
      float ac = d[0] - l, duc = e[0], bc = z[0];
      float lo = duc, dn = d[1], en = e[1], bn = z[min(1, c - 1) * ldz];
#pragma unroll 1
      for (int j = 0; j + 1 < c; ++j) {
        // the next row's entries, before the stores
        const float d2 = d[j + 2], e2 = e[j + 2], b2 = z[min(j + 2, c - 1) * ldz];
        const float an = dn - l, dun = en;
        const bool keep = fabsf(ac) >= fabsf(lo);
        const float piv = keep ? (ac == 0.0f ? tiny : ac) : lo;
        const float f = __uint_as_float((__float_as_uint(__fdividef(keep ? lo : ac, piv)) & ~1u) | keep);
        rp[j * ldf] = __fdividef(1.0f, fabsf(piv) < tiny ? copysignf(tiny, piv) : piv);
        du[j * ldf] = keep ? duc : an;
        du2[j * ldf] = keep ? 0.0f : dun;
        fm[j * ldf] = f;
        z[j * ldz] = keep ? bc : bn;
        const float na = keep ? fmaf(-f, duc, an) : fmaf(-f, an, duc);
        const float nd = keep ? dun : -f * dun;
        const float nbv = keep ? fmaf(-f, bc, bn) : fmaf(-f, bn, bc);
        ac = na;
        duc = nd;
        bc = nbv;
        lo = en;
        dn = d2;
        en = e2;
        bn = b2;
      }
      rp[(c - 1) * ldf] = __fdividef(1.0f, fabsf(ac) < tiny ? copysignf(tiny, ac) : ac);
      du[(c - 1) * ldf] = 0.0f;
      du2[(c - 1) * ldf] = 0.0f;
      z[(c - 1) * ldz] = bc;
      back_solve(z, ldz, rp, du, du2, ldf, c);
    }
#pragma unroll 1
    for (int it = 0; it < 2; ++it) {
      __syncthreads();
      // unit length, a warp per vector: by the largest entry first (the square
      // may overflow)
      for (int i2 = i0 + warp; i2 < min(c, i0 + nb); i2 += kW) {
        float zr[CT], mx = 0.0f, s = 0.0f;
#pragma unroll
        for (int t = 0; t < CT; ++t) {
          const int r = lane + 32 * t;
          zr[t] = r < c ? Z[r * ldz + i2] : 0.0f;
          mx = fmaxf(mx, fabsf(zr[t]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        const float s1 = mx > 0.0f ? 1.0f / mx : 0.0f;
#pragma unroll
        for (int t = 0; t < CT; ++t) {
          zr[t] *= s1;
          s = fmaf(zr[t], zr[t], s);
        }
        s = warp_sum(s);
        const float inv = s > 0.0f ? rsqrtf(s) : 0.0f;
#pragma unroll
        for (int t = 0; t < CT; ++t)
          if (lane + 32 * t < c) Z[(lane + 32 * t) * ldz + i2] = zr[t] * inv;
      }
      __syncthreads();
      if (it == 0 && on) {               // second step: the kept factors
        float bc = z[0], bn = z[min(1, c - 1) * ldz], f = fm[0];
#pragma unroll 1
        for (int j = 0; j + 1 < c; ++j) {
          const int j2 = min(j + 2, c - 1);
          const float bn2 = z[j2 * ldz], f2 = fm[(j2 - 1) * ldf];
          const bool keep = __float_as_uint(f) & 1u;
          z[j * ldz] = keep ? bc : bn;
          bc = keep ? fmaf(-f, bc, bn) : fmaf(-f, bn, bc);
          bn = bn2;
          f = f2;
        }
        z[(c - 1) * ldz] = bc;
        back_solve(z, ldz, rp, du, du2, ldf, c);
      }
    }
  }

  // 4. Gram-Schmidt inside clusters: lam decreasing, a new cluster where the gap
  // exceeds the threshold. s_end[i]: one past the cluster of i; s_list: the
  // vectors that have later ones in their cluster, in order.
  if (warp == 0) {
    int n = 0;
    for (int i0 = 0; i0 < c; i0 += 32) {
      const int i = i0 + lane;
      const bool last = i >= c - 1 || lam[i] - lam[i + 1] > kClusterRel * span;
      const unsigned m = __ballot_sync(0xffffffffu, i < c && !last);
      if (i < c && !last) s_list[n + __popc(m & ((1u << lane) - 1u))] = i;
      if (i < c) s_end[i] = last ? i + 1 : 0;
      n += __popc(m);
    }
    __syncwarp();
    if (lane == 0) {
      s_count = n;
      for (int i = c - 2; n > 0 && i >= 0; --i)
        if (s_end[i] == 0) s_end[i] = s_end[i + 1];
    }
  }
  __syncthreads();
  if (s_count > 0) {
    float z[R][CT];                      // vector warp + 16 q in z[q]
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
      for (int t = 0; t < CT; ++t) {
        const int r = lane + 32 * t, i = warp + kW * q;
        z[q][t] = (r < c && i < c) ? Z[r * ldz + i] : 0.0f;
      }
    auto finish = [&](auto which, float *buf, int sweep) {
      constexpr int q = decltype(which)::value;
      float s = 0.0f;
#pragma unroll
      for (int t = 0; t < CT; ++t) s = fmaf(z[q][t], z[q][t], s);
      s = warp_sum(s);
      if (s < 0.5f && sweep == 0 && lane == 0) s_again = 1;
      const float inv = s > 0.0f ? rsqrtf(s) : 0.0f;
#pragma unroll
      for (int t = 0; t < CT; ++t) {
        z[q][t] *= inv;
        buf[lane + 32 * t] = z[q][t];
      }
    };
#pragma unroll 1
    for (int sweep = 0; sweep < 2; ++sweep) {
#pragma unroll 1
      for (int n = 0; n <= s_count; ++n) {
        // finish vector ai (its warp): unit length, to shared memory. After the
        // last listed vector only that vector's successor remains, in every
        // cluster; they are scaled below.
        const int ai = n < s_count ? s_list[n] : -1;
        float *buf = s_zb[n & 1];
        if (ai >= 0 && warp == ai % kW) {
          switch (ai / kW) {
            case 0: finish(std::integral_constant<int, 0>{}, buf, sweep); break;
            case 1: finish(std::integral_constant<int, 1>{}, buf, sweep); break;
            case 2: finish(std::integral_constant<int, 2>{}, buf, sweep); break;
            case 3: finish(std::integral_constant<int, 3>{}, buf, sweep); break;
            case 4: finish(std::integral_constant<int, R == 8 ? 4 : 0>{}, buf, sweep); break;
            case 5: finish(std::integral_constant<int, R == 8 ? 5 : 0>{}, buf, sweep); break;
            case 6: finish(std::integral_constant<int, R == 8 ? 6 : 0>{}, buf, sweep); break;
            default: finish(std::integral_constant<int, R == 8 ? 7 : 0>{}, buf, sweep); break;
          }
        }
        if (ai < 0) break;
        __syncthreads();
        float x[CT], acc[R];
#pragma unroll
        for (int t = 0; t < CT; ++t) x[t] = buf[lane + 32 * t];
        const int end = s_end[ai];
#pragma unroll
        for (int q = 0; q < R; ++q) {
          acc[q] = z[q][0] * x[0];
#pragma unroll
          for (int t = 1; t < CT; ++t) acc[q] = fmaf(z[q][t], x[t], acc[q]);
        }
        const float s = warp_sums<R>(acc, lane);
#pragma unroll
        for (int q = 0; q < R; ++q) {
          // lane that holds the sum of value q
          const int src = R == 8 ? ((q >> 2) & 1) * 16 + ((q >> 1) & 1) * 8 + (q & 1) * 4
                                 : ((q >> 1) & 1) * 16 + (q & 1) * 8;
          const float dot = __shfl_sync(0xffffffffu, s, src);
          const int i = warp + kW * q;
          if (i > ai && i < end) {
#pragma unroll
            for (int t = 0; t < CT; ++t) z[q][t] = fmaf(-dot, x[t], z[q][t]);
          }
        }
      }
      // every vector to unit length (the last ones of the clusters have not been)
#pragma unroll
      for (int q = 0; q < R; ++q) {
        float s = 0.0f;
#pragma unroll
        for (int t = 0; t < CT; ++t) s = fmaf(z[q][t], z[q][t], s);
        s = warp_sum(s);
        if (s < 0.5f && warp + kW * q < c && sweep == 0 && lane == 0) s_again = 1;
        const float inv = s > 0.0f ? rsqrtf(s) : 0.0f;
#pragma unroll
        for (int t = 0; t < CT; ++t) z[q][t] *= inv;
      }
      __syncthreads();
      if (!s_again) break;
    }
#pragma unroll
    for (int q = 0; q < R; ++q)
#pragma unroll
      for (int t = 0; t < CT; ++t) {
        const int r = lane + 32 * t, i = warp + kW * q;
        if (r < c && i < c) Z[r * ldz + i] = z[q][t];
      }
    __syncthreads();
  }

  // 5. back-transformation Z <- H_0 ... H_{c-3} Z: four lanes per column, lane s
  // holds rows 16 t + 4 s .. + 3 (two columns per quad: 60% slower)
  if (warp * 8 < c) {
    constexpr int NT4 = 2 * CT;
    const int i = tid >> 2, s = tid & 3;
    float z[NT4][4];
#pragma unroll
    for (int t = 0; t < NT4; ++t)
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int r = 16 * t + 4 * s + m;
        z[t][m] = (r < c && i < c) ? Z[r * ldz + i] : 0.0f;
      }
#pragma unroll 1
    for (int k = c - 3; k >= 0; --k) {
      const float beta = tau[k];
      if (beta == 0.0f) continue;
      const int t0 = (k + 1) >> 4;       // rows below 16 t0 are zero in v
      const float4 *v = reinterpret_cast<const float4 *>(Vh + k * LDV) + s;
      float4 vr[NT4];
      float dot0 = 0.0f, dot1 = 0.0f;
#pragma unroll
      for (int t = 0; t < NT4; ++t)
        if (t >= t0) {
          vr[t] = v[4 * t];
          dot0 = fmaf(vr[t].x, z[t][0], fmaf(vr[t].y, z[t][1], dot0));
          dot1 = fmaf(vr[t].z, z[t][2], fmaf(vr[t].w, z[t][3], dot1));
        }
      float dot = dot0 + dot1;
      dot += __shfl_xor_sync(0xffffffffu, dot, 1);
      dot += __shfl_xor_sync(0xffffffffu, dot, 2);
      const float f = -beta * dot;
#pragma unroll
      for (int t = 0; t < NT4; ++t)
        if (t >= t0) {
          z[t][0] = fmaf(f, vr[t].x, z[t][0]);
          z[t][1] = fmaf(f, vr[t].y, z[t][1]);
          z[t][2] = fmaf(f, vr[t].z, z[t][2]);
          z[t][3] = fmaf(f, vr[t].w, z[t][3]);
        }
    }
#pragma unroll
    for (int t = 0; t < NT4; ++t)
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        const int r = 16 * t + 4 * s + m;
        if (r < c && i < c) Z[r * ldz + i] = z[t][m];
      }
  }
  __syncthreads();
  for (int r = warp; r < c; r += kW)
    for (int i = lane; i < c; i += 32) U[r * c + i] = to_f64(Z[r * ldz + i]);
}

template <int CT>
cudaError_t launch_start(const double *G, int c, double *U, const int *skip, cudaStream_t st) {
  const size_t smem = eig_smem<CT>(c);
  const cudaError_t e = cudaFuncSetAttribute(eig_start_kernel<CT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             (int)eig_smem<CT>(32 * CT));
  if (e != cudaSuccess) return e;
  launch_k(eig_start_kernel<CT>, 1, kT, smem, st, G, c, U, skip);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

cudaError_t eig_start(const double *G, int c, double *U, const int *skip, cudaStream_t st) {
  if (c < 1 || c > kMaxSmall) return cudaErrorInvalidValue;
  if (c <= 64) return launch_start<2>(G, c, U, skip, st);
  if (c <= 96) return launch_start<3>(G, c, U, skip, st);
  return launch_start<4>(G, c, U, skip, st);
}

}  // namespace hatt
