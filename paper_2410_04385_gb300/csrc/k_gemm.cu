// Batched, arbitrarily strided FP64 GEMM for the small contractions of HaTT.
//
// On GB300 the FP64 pipe delivers ~1.2 TFLOP/s, about two DFMA lanes per SM
// per clock, against ~73 TFLOP/s of FP32. A warp-wide DFMA therefore occupies
// the SM's FP64 unit for ~16 clocks while the two shared-memory operand loads
// it needs take ~3 wavefronts: an FP64 contraction is bound by DFMA issue, and
// register blocking buys nothing. What costs time is every DFMA a warp issues
// for an output slot that some of its lanes do not have -- a predicated-off
// DFMA holds the FP64 unit as long as a full one (ncu: a 625-output tile dealt
// as four slots per thread kept the pipe busy for 32 warp-DFMAs per k step
// where 20 carry outputs) -- and every idle SM. So:
//   * a block computes a bm x bn output tile of any shape (bm, bn <= 128,
//     bm*bn <= 4096), its outputs dealt linearly to 256 threads; each warp
//     runs the multiply-add loop for exactly the number of slots its lane 0
//     owns (a warp-uniform switch, no predicated-off slots), and tiles are
//     chosen by a cost model that counts those warp-DFMAs, so almost no DFMA
//     is spent on padding;
//   * K is split until the grid has about four blocks per SM (wave
//     quantization < 25%); the block that finishes an output tile last (a
//     per-tile counter) sums its split-K partials in split order 0..ksplit-1,
//     whichever block that is, so results are bitwise reproducible and no
//     second kernel is launched.
#include <algorithm>
#include <unordered_map>
#include <array>
#include <cstdlib>
#include <cstring>
#include <atomic>
#include <mutex>
#include <type_traits>
#include <vector>
#include "hatt_internal.cuh"

namespace hatt {
namespace {

constexpr int kBK = 16;
constexpr int kThreads = 256;
constexpr int kMaxTile = 128;            // bm, bn <= kMaxTile
constexpr int kMaxOut = 16;              // outputs per thread -> bm*bn <= 4096
constexpr int kTargetBlocks = 4 * 152;

struct Launch {
  int bm, bn, tiles_m, tiles_n, ksplit, kchunk, out;
  bool pair = false;                     // gemm_pair_kernel: slots of two adjacent columns
};

// Operand of a low-precision product: FP64 -> FP32 (round to nearest even),
// then, for TF32, round to nearest with ties away from zero at 10 mantissa
// bits, and for BF16 round to nearest even at 7 mantissa bits: the values a
// tensor core multiplies (exactly) and accumulates in FP32.
__device__ __forceinline__ float round_operand(double x, int prec) {
  const float f = (float)x;
  unsigned u = __float_as_uint(f);
  if (prec == kPrecTF32) u = (u + 0x1000u) & 0xFFFFE000u;
  else if (prec == kPrecBF16) u = (u + 0x7FFFu + ((u >> 16) & 1u)) & 0xFFFF0000u;
  return __uint_as_float(u);
}

// acc[q] += sum over the k slice of As[k][om[q]] Bs[k][on[q]] for the first NQ
// output slots. Lanes that own fewer slots than NQ multiply valid shared-memory
// entries (their indices are 0) into accumulators that are never stored.
template <int NQ, int OUT, typename T>
__device__ __forceinline__ void mac_n(int kdepth, const T (*As)[kMaxTile + 1],
                                      const T (*Bs)[kMaxTile + 1], const int (&om)[OUT],
                                      const int (&on)[OUT], T (&acc)[OUT]) {
  if (kdepth == kBK) {
#pragma unroll 4
    for (int kk = 0; kk < kBK; ++kk) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) acc[q] = fma(As[kk][om[q]], Bs[kk][on[q]], acc[q]);
    }
  } else {
    for (int kk = 0; kk < kdepth; ++kk) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) acc[q] = fma(As[kk][om[q]], Bs[kk][on[q]], acc[q]);
    }
  }
}

// Dispatch on the warp-uniform slot count nqw in [0, OUT].
template <int NQ, int OUT, typename T>
__device__ __forceinline__ void mac_slots(int nqw, int kdepth, const T (*As)[kMaxTile + 1],
                                          const T (*Bs)[kMaxTile + 1], const int (&om)[OUT],
                                          const int (&on)[OUT], T (&acc)[OUT]) {
  if (nqw <= 0) return;
  if (nqw == NQ) {
    mac_n<NQ, OUT, T>(kdepth, As, Bs, om, on, acc);
    return;
  }
  if constexpr (NQ < OUT) mac_slots<NQ + 1, OUT, T>(nqw, kdepth, As, Bs, om, on, acc);
}

// Live column count and depth of a product whose extents depend on a rank in
// device memory (Gemm::dyn_dev); the planned (g.N, g.K) otherwise.
__device__ __forceinline__ void live_extents(const Gemm &g, int &N, int &K) {
  N = g.N;
  K = g.K;
  if (g.dyn_dev == nullptr) return;
  const long long R = max(*g.dyn_dev, 0);
  if (g.dyn_n > 0) N = (int)min((long long)N, g.dyn_n * R);
  if (g.dyn_k > 0) K = (int)min((long long)K, g.dyn_k * R);
}

// LOWP = false: FP64 operands and accumulators. LOWP = true: operands rounded
// to g.prec as they are staged (above) and FP32 accumulators; the result is
// written in FP64 (scaled by alpha in FP64).
template <int OUT, bool LOWP>
__global__ void __launch_bounds__(kThreads)
gemm_f64_kernel(Gemm g, int bm, int bn, int tiles_n, int tiles_m, int ksplit, int kchunk,
                double *partial, int *counters) {
  pdl_enter();
  using T = typename std::conditional<LOWP, float, double>::type;
  if (g.skip_dev && *g.skip_dev) return;
  __shared__ T As[kBK][kMaxTile + 1];
  __shared__ T Bs[kBK][kMaxTile + 1];
  __shared__ int s_last;
  const int prec = g.prec;
  const int tid = threadIdx.x;
  // 1-D grid: block -> (n tile, m tile, split, batch), n tile fastest
  long long blk = blockIdx.x;
  const int tn_i = (int)(blk % tiles_n); blk /= tiles_n;
  const int tm_i = (int)(blk % tiles_m); blk /= tiles_m;
  const int ks = (int)(blk % ksplit);
  const int b = (int)(blk / ksplit);
  const int b1 = b / g.bdiv, b2 = b % g.bdiv;
  const double *A = g.A + b1 * g.sA1 + b2 * g.sA2;
  const double *B = g.B + b1 * g.sB1 + b2 * g.sB2;
  const int m0 = tm_i * bm, n0 = tn_i * bn;
  int N, K;
  live_extents(g, N, K);
  if (n0 >= N) return;   // a tile past the live columns: every K split of it leaves here
  const int kbeg = ks * kchunk;
  const int kend = min(K, kbeg + kchunk);
  const int outs = bm * bn;

  int om[OUT], on[OUT];
  T acc[OUT];
#pragma unroll
  for (int q = 0; q < OUT; ++q) {
    const int o = tid + kThreads * q;
    om[q] = (o < outs) ? o / bn : 0;
    on[q] = (o < outs) ? o % bn : 0;
    acc[q] = 0.0;
  }
  const int nq = (outs - tid + kThreads - 1) / kThreads;   // outputs this thread owns
  // lane 0 owns the most outputs of its warp (nq does not increase with tid)
  const int nqw = __shfl_sync(0xffffffffu, nq, 0);

  const bool a_kfast = (g.sAk == 1);
  const bool b_nfast = (g.sBn == 1);
  for (int kt = kbeg; kt < kend; kt += kBK) {
    for (int e = tid; e < bm * kBK; e += kThreads) {
      int mm, kk;
      if (a_kfast) { mm = e / kBK; kk = e % kBK; } else { kk = e / bm; mm = e % bm; }
      const int gm = m0 + mm, gk = kt + kk;
      const double v = (gm < g.M && gk < kend) ? A[gm * g.sAm + gk * g.sAk] : 0.0;
      if (LOWP) As[kk][mm] = round_operand(v, prec); else As[kk][mm] = v;
    }
    for (int e = tid; e < bn * kBK; e += kThreads) {
      int nn, kk;
      if (b_nfast) { kk = e / bn; nn = e % bn; } else { nn = e / kBK; kk = e % kBK; }
      const int gn = n0 + nn, gk = kt + kk;
      const double v = (gn < N && gk < kend) ? B[gk * g.sBk + gn * g.sBn] : 0.0;
      if (LOWP) Bs[kk][nn] = round_operand(v, prec); else Bs[kk][nn] = v;
    }
    __syncthreads();
    // exact depth: a ragged last k-tile issues no DFMAs on zero padding
    mac_slots<1, OUT>(nqw, min(kBK, kend - kt), As, Bs, om, on, acc);
    __syncthreads();
  }

  const double alpha = g.alpha * (g.alpha_dev ? *g.alpha_dev : 1.0);
  double *C = g.C + b1 * g.sC1 + b2 * g.sC2;
  if (ksplit > 1) {
    const long long mn = (long long)g.M * g.N;
    const double *P0 = partial + (long long)b * ksplit * mn;
    double *P = partial + ((long long)b * ksplit + ks) * mn;
#pragma unroll
    for (int q = 0; q < OUT; ++q) {
      if (q >= nq) break;
      const int gm = m0 + om[q], gn = n0 + on[q];
      if (gm < g.M && gn < N) P[(long long)gm * g.N + gn] = (double)acc[q];
    }
    // publish this partial, then let the last of the tile's ksplit blocks sum
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      const int t = (b * tiles_m + tm_i) * tiles_n + tn_i;
      const int prev = atomicAdd(&counters[t], 1);
      s_last = (prev == ksplit - 1);
      if (s_last) counters[t] = 0;          // clean for the next GEMM on this array
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll
    for (int q = 0; q < OUT; ++q) {
      if (q >= nq) break;
      const int gm = m0 + om[q], gn = n0 + on[q];
      if (gm >= g.M || gn >= N) continue;
      const long long e = (long long)gm * g.N + gn;
      double sum = 0.0;
      for (int k = 0; k < ksplit; ++k) sum += (k == ks) ? (double)acc[q] : __ldcg(P0 + k * mn + e);
      double *c = C + gm * g.sCm + gn * g.sCn;
      const double v = alpha * sum;
      *c = (g.beta != 0.0) ? fma(g.beta, *c, v) : v;
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < OUT; ++q) {
    if (q >= nq) break;
    const int gm = m0 + om[q], gn = n0 + on[q];
    if (gm >= g.M || gn >= N) continue;
    double *c = C + gm * g.sCm + gn * g.sCn;
    const double v = alpha * (double)acc[q];
    *c = (g.beta != 0.0) ? fma(g.beta, *c, v) : v;
  }
}

// Pair variant (FP64 only): an output slot is a row and two adjacent columns,
// so one shared-memory load of A and one 16-byte load of B feed two DFMAs
// (one and a half loads per DFMA against two). On the short-K batched
// products of the sweep it is the faster form; on long split-K products the
// single form is. Which one a shape runs is decided by timing (exec_plan). Only
// calls that keep their arithmetic (set_kept_arithmetic) run it: elsewhere the
// products it was made for go to the tensor cores (k_gemm_split.cu).
constexpr int kLdB2 = kMaxTile + 2;      // even row stride: 16-byte aligned B rows

template <int NQ, int OUT>
__device__ __forceinline__ void mac_pair_n(int kdepth, const double (*As)[kMaxTile + 1],
                                           const double (*Bs)[kLdB2], const int (&om)[OUT],
                                           const int (&on)[OUT], double (&a0)[OUT],
                                           double (&a1)[OUT]) {
  if (kdepth == kBK) {
#pragma unroll 4
    for (int kk = 0; kk < kBK; ++kk) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const double a = As[kk][om[q]];
        const double2 bb = *reinterpret_cast<const double2 *>(&Bs[kk][on[q]]);
        a0[q] = fma(a, bb.x, a0[q]);
        a1[q] = fma(a, bb.y, a1[q]);
      }
    }
  } else {
    for (int kk = 0; kk < kdepth; ++kk) {
#pragma unroll
      for (int q = 0; q < NQ; ++q) {
        const double a = As[kk][om[q]];
        const double2 bb = *reinterpret_cast<const double2 *>(&Bs[kk][on[q]]);
        a0[q] = fma(a, bb.x, a0[q]);
        a1[q] = fma(a, bb.y, a1[q]);
      }
    }
  }
}

template <int NQ, int OUT>
__device__ __forceinline__ void mac_pair_slots(int nqw, int kdepth, const double (*As)[kMaxTile + 1],
                                               const double (*Bs)[kLdB2], const int (&om)[OUT],
                                               const int (&on)[OUT], double (&a0)[OUT],
                                               double (&a1)[OUT]) {
  if (nqw <= 0) return;
  if (nqw == NQ) {
    mac_pair_n<NQ, OUT>(kdepth, As, Bs, om, on, a0, a1);
    return;
  }
  if constexpr (NQ < OUT) mac_pair_slots<NQ + 1, OUT>(nqw, kdepth, As, Bs, om, on, a0, a1);
}

template <int OUT>
__global__ void __launch_bounds__(kThreads)
gemm_pair_kernel(Gemm g, int bm, int bn, int tiles_n, int tiles_m, int ksplit, int kchunk,
                 double *partial, int *counters) {
  pdl_enter();
  if (g.skip_dev && *g.skip_dev) return;
  __shared__ double As[kBK][kMaxTile + 1];
  __shared__ __align__(16) double Bs[kBK][kLdB2];
  __shared__ int s_last;
  const int tid = threadIdx.x;
  long long blk = blockIdx.x;
  const int tn_i = (int)(blk % tiles_n); blk /= tiles_n;
  const int tm_i = (int)(blk % tiles_m); blk /= tiles_m;
  const int ks = (int)(blk % ksplit);
  const int b = (int)(blk / ksplit);
  const int b1 = b / g.bdiv, b2 = b % g.bdiv;
  const double *A = g.A + b1 * g.sA1 + b2 * g.sA2;
  const double *B = g.B + b1 * g.sB1 + b2 * g.sB2;
  const int m0 = tm_i * bm, n0 = tn_i * bn;
  int N, K;
  live_extents(g, N, K);
  if (n0 >= N) return;   // a tile past the live columns: every K split of it leaves here
  const int kbeg = ks * kchunk;
  const int kend = min(K, kbeg + kchunk);
  const int bn2 = (bn + 1) / 2, bnp = 2 * bn2;   // column pairs; an odd tail column pairs with zero
  const int slots = bm * bn2;

  int om[OUT], on[OUT];
  double a0[OUT], a1[OUT];
#pragma unroll
  for (int q = 0; q < OUT; ++q) {
    const int o = tid + kThreads * q;
    om[q] = (o < slots) ? o / bn2 : 0;
    on[q] = (o < slots) ? 2 * (o % bn2) : 0;
    a0[q] = 0.0;
    a1[q] = 0.0;
  }
  const int nq = (slots - tid + kThreads - 1) / kThreads;
  const int nqw = __shfl_sync(0xffffffffu, nq, 0);

  const bool a_kfast = (g.sAk == 1);
  const bool b_nfast = (g.sBn == 1);
  for (int kt = kbeg; kt < kend; kt += kBK) {
    for (int e = tid; e < bm * kBK; e += kThreads) {
      int mm, kk;
      if (a_kfast) { mm = e / kBK; kk = e % kBK; } else { kk = e / bm; mm = e % bm; }
      const int gm = m0 + mm, gk = kt + kk;
      As[kk][mm] = (gm < g.M && gk < kend) ? A[gm * g.sAm + gk * g.sAk] : 0.0;
    }
    for (int e = tid; e < bnp * kBK; e += kThreads) {
      int nn, kk;
      if (b_nfast) { kk = e / bnp; nn = e % bnp; } else { nn = e / kBK; kk = e % kBK; }
      const int gn = n0 + nn, gk = kt + kk;
      Bs[kk][nn] = (nn < bn && gn < N && gk < kend) ? B[gk * g.sBk + gn * g.sBn] : 0.0;
    }
    __syncthreads();
    mac_pair_slots<1, OUT>(nqw, min(kBK, kend - kt), As, Bs, om, on, a0, a1);
    __syncthreads();
  }

  const double alpha = g.alpha * (g.alpha_dev ? *g.alpha_dev : 1.0);
  double *C = g.C + b1 * g.sC1 + b2 * g.sC2;
  if (ksplit > 1) {
    const long long mn = (long long)g.M * g.N;
    const double *P0 = partial + (long long)b * ksplit * mn;
    double *P = partial + ((long long)b * ksplit + ks) * mn;
#pragma unroll
    for (int q = 0; q < OUT; ++q) {
      if (q >= nq) break;
      const int gm = m0 + om[q], gn = n0 + on[q];
      if (gm >= g.M) continue;
      if (on[q] < bn && gn < N) P[(long long)gm * g.N + gn] = a0[q];
      if (on[q] + 1 < bn && gn + 1 < N) P[(long long)gm * g.N + gn + 1] = a1[q];
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) {
      const int t = (b * tiles_m + tm_i) * tiles_n + tn_i;
      const int prev = atomicAdd(&counters[t], 1);
      s_last = (prev == ksplit - 1);
      if (s_last) counters[t] = 0;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll
    for (int q = 0; q < OUT; ++q) {
      if (q >= nq) break;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int gm = m0 + om[q], gn = n0 + on[q] + h;
        if (gm >= g.M || on[q] + h >= bn || gn >= N) continue;
        const long long e = (long long)gm * g.N + gn;
        const double own = h ? a1[q] : a0[q];
        double sum = 0.0;
        for (int k = 0; k < ksplit; ++k) sum += (k == ks) ? own : __ldcg(P0 + k * mn + e);
        double *c = C + gm * g.sCm + gn * g.sCn;
        const double v = alpha * sum;
        *c = (g.beta != 0.0) ? fma(g.beta, *c, v) : v;
      }
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < OUT; ++q) {
    if (q >= nq) break;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int gm = m0 + om[q], gn = n0 + on[q] + h;
      if (gm >= g.M || on[q] + h >= bn || gn >= N) continue;
      double *c = C + gm * g.sCm + gn * g.sCn;
      const double v = alpha * (h ? a1[q] : a0[q]);
      *c = (g.beta != 0.0) ? fma(g.beta, *c, v) : v;
    }
  }
}

long long ceil_div(long long a, long long b) { return (a + b - 1) / b; }

// Tile edge for a dimension X with edge cap `cap`: X itself if it fits, else
// the edge in [cap/2, cap] with the least padding (larger on ties).
int tile_edge(int X, int cap) {
  if (X <= cap) return X;
  int best = cap;
  long long best_pad = ceil_div(X, cap) * cap;
  for (int t = cap - 1; t >= std::max(1, cap / 2); --t) {
    const long long pad = ceil_div(X, t) * t;
    if (pad < best_pad) {
      best_pad = pad;
      best = t;
    }
  }
  return best;
}

// Warp-DFMA clocks per k step of one block: each warp issues one DFMA per
// output slot its lane 0 owns, and a warp-DFMA holds the SM's FP64 unit
// (two lanes per clock) for 16 clocks.
double block_dfma_clocks(long long outs) {
  double warp_slots = 0.0;
  for (int w = 0; w < kThreads / 32; ++w)
    warp_slots += (double)std::max<long long>(0, ceil_div(outs - 32LL * w, kThreads));
  return 16.0 * warp_slots;
}

int out_slots(long long outs) {
  const long long need = ceil_div(outs, kThreads);
  return need <= 1 ? 1 : need <= 2 ? 2 : need <= 4 ? 4 : need <= 8 ? 8 : need <= 12 ? 12 : 16;
}

// Analytic launch model (clocks of the busiest SM) used to pick the tile and
// the K split:
//   FP64: the warp-DFMAs of a block (block_dfma_clocks per k step) times the
//         number of blocks the busiest SM receives (wave quantization over
//         152 SMs);
//   latency: ~450 clocks per 16-deep k-tile (staging + two barriers), hidden
//         by the blocks resident on an SM (fewer when a thread holds more
//         accumulators);
//   split-K: the last block of each tile re-reads the tile's ksplit partial
//         sums from L2 (~64 bytes per clock per SM) before it writes C; the
//         busiest SM does ceil(tiles / 152) such reductions.
double model_clocks(const Gemm &g, int bm, int bn, long long ksplit, bool pair = false) {
  const long long tiles = ceil_div(g.M, bm) * ceil_div(g.N, bn) * (long long)g.batch;
  const long long kchunk = ceil_div(ceil_div(g.K, ksplit), kBK) * kBK;
  const long long nsplit = ceil_div(g.K, kchunk);
  const long long blocks = tiles * nsplit;
  const long long per_sm = ceil_div(blocks, 152);
  const long long kdepth = std::min<long long>(kchunk, g.K);
  const long long outs = (long long)bm * bn;
  const long long slots = pair ? (long long)bm * ((bn + 1) / 2) : outs;
  const int out = out_slots(slots);
  const int resident = out <= 4 ? 4 : out <= 8 ? 3 : 2;
  const double ktiles = (double)ceil_div(kdepth, kBK);
  double t = per_sm * (double)kdepth * block_dfma_clocks(slots) * (pair ? 2.0 : 1.0) +
             ceil_div(per_sm, resident) * ktiles * 450.0 + 1500.0;
  if (nsplit > 1)
    t += (double)ceil_div(tiles, 152) * (600.0 + (double)nsplit * outs * 8.0 / 64.0);
  return t;
}

// Candidate tile edges for a dimension X: every divisor of X up to
// kMaxTile, and the least-padding edge below each power-of-two cap.
int edge_candidates(int X, int *out) {
  int n = 0;
  for (int t = 1; t <= std::min(X, kMaxTile); ++t)
    if (X % t == 0) out[n++] = t;
  static const int caps[5] = {128, 64, 32, 16, 8};
  for (int cap : caps) {
    const int t = tile_edge(X, cap);
    bool have = false;
    for (int i = 0; i < n; ++i) have |= (out[i] == t);
    if (!have) out[n++] = t;
  }
  return n;
}

// Normalizes a (bm, bn, ksplit) choice: tile counts, output slots per
// thread, the K chunk and the number of K slices that chunk gives.
Launch finalize(const Gemm &g, int bm, int bn, long long ksplit, bool pair) {
  Launch L{};
  L.bm = bm;
  L.bn = bn;
  L.pair = pair;
  L.tiles_m = (int)ceil_div(g.M, bm);
  L.tiles_n = (int)ceil_div(g.N, bn);
  L.out = out_slots(pair ? (long long)bm * ((bn + 1) / 2) : (long long)bm * bn);
  const long long kchunk = ceil_div(ceil_div(g.K, ksplit), kBK) * kBK;
  L.kchunk = (int)std::max<long long>(kchunk, kBK);
  L.ksplit = (int)ceil_div(g.K, L.kchunk);
  return L;
}

// Every (tile, K split) candidate with its model clocks, single or pair form.
void plan_candidates(const Gemm &g, bool pair, std::vector<std::pair<double, Launch>> &out) {
  int em[kMaxTile + 8], en[kMaxTile + 8];
  const int nm = edge_candidates(g.M, em), nn = edge_candidates(g.N, en);
  for (int j = 0; j < nn; ++j) {
    const int bn = en[j];
    for (int i = 0; i < nm; ++i) {
      const int bm = em[i];
      const long long slots = pair ? (long long)bm * ((bn + 1) / 2) : (long long)bm * bn;
      if (slots > (long long)kThreads * (pair ? 8 : kMaxOut)) continue;
      if (pair && bn < 2) continue;
      const long long tiles = ceil_div(g.M, bm) * ceil_div(g.N, bn) * (long long)g.batch;
      const long long kmax = ceil_div(g.K, kBK);
      long long cands[12];
      int nc = 0;
      for (long long s = 1; s <= kmax && nc < 10; s *= 2) cands[nc++] = s;
      cands[nc++] = std::min(kmax, std::max<long long>(1, ceil_div(kTargetBlocks, tiles)));
      cands[nc++] = std::min(kmax, std::max<long long>(1, ceil_div(152, tiles)));
      for (int c = 0; c < nc; ++c) {
        if (cands[c] > 1 && tiles > kTileCounters) continue;   // one counter per tile
        out.push_back({model_clocks(g, bm, bn, cands[c], pair), finalize(g, bm, bn, cands[c], pair)});
      }
    }
  }
}

Launch plan_search(const Gemm &g) {
  std::vector<std::pair<double, Launch>> c;
  plan_candidates(g, false, c);
  double best = 1e300;
  Launch L{};
  for (const auto &x : c)
    if (x.first < best) {
      best = x.first;
      L = x.second;
    }
  return L;
}

// Plans are cached per shape in hash maps: launch-bound callers (power
// iteration, small eager recompressions) look a plan up for every GEMM, and a
// batch of uneven pairs brings thousands of shapes.
struct ShapeHash {
  size_t operator()(const std::array<int, 8> &k) const {
    size_t h = 1469598103934665603ull;
    for (int v : k) h = (h ^ (size_t)(unsigned)v) * 1099511628211ull;
    return h;
  }
};
using ShapeKey = std::array<int, 8>;

Launch plan(const Gemm &g) {
  static std::mutex mu;
  static std::unordered_map<ShapeKey, Launch, ShapeHash> cache;
  const ShapeKey key{g.M, g.N, g.K, g.batch, 0, 0, 0, 0};
  {
    std::lock_guard<std::mutex> lock(mu);
    const auto it = cache.find(key);
    if (it != cache.end()) return it->second;
  }
  const Launch L = plan_search(g);
  std::lock_guard<std::mutex> lock(mu);
  if (cache.size() < (1u << 16)) cache.emplace(key, L);
  return L;
}

template <int OUT>
void launch_tile(const Gemm &g, const Launch &L, double *scratch, int *counters,
                 cudaStream_t st) {
  const long long blocks = (long long)L.tiles_n * L.tiles_m * L.ksplit * g.batch;
  if (g.prec == kPrecFP64)
    launch_k(gemm_f64_kernel<OUT, false>, (unsigned)blocks, kThreads, 0, st, 
        g, L.bm, L.bn, L.tiles_n, L.tiles_m, L.ksplit, L.kchunk, scratch, counters);
  else
    launch_k(gemm_f64_kernel<OUT, true>, (unsigned)blocks, kThreads, 0, st, 
        g, L.bm, L.bn, L.tiles_n, L.tiles_m, L.ksplit, L.kchunk, scratch, counters);
  note_launch();
}

template <int OUT>
void launch_pair(const Gemm &g, const Launch &L, double *scratch, int *counters, cudaStream_t st) {
  const long long blocks = (long long)L.tiles_n * L.tiles_m * L.ksplit * g.batch;
  launch_k(gemm_pair_kernel<OUT>, (unsigned)blocks, kThreads, 0, st,
      g, L.bm, L.bn, L.tiles_n, L.tiles_m, L.ksplit, L.kchunk, scratch, counters);
  note_launch();
}

void launch_plan(const Gemm &g, const Launch &L, double *scratch, int *counters, cudaStream_t st) {
  if (L.pair) {
    switch (L.out) {
      case 1: launch_pair<1>(g, L, scratch, counters, st); break;
      case 2: launch_pair<2>(g, L, scratch, counters, st); break;
      case 4: launch_pair<4>(g, L, scratch, counters, st); break;
      default: launch_pair<8>(g, L, scratch, counters, st); break;
    }
    return;
  }
  switch (L.out) {
    case 1: launch_tile<1>(g, L, scratch, counters, st); break;
    case 2: launch_tile<2>(g, L, scratch, counters, st); break;
    case 4: launch_tile<4>(g, L, scratch, counters, st); break;
    case 8: launch_tile<8>(g, L, scratch, counters, st); break;
    case 12: launch_tile<12>(g, L, scratch, counters, st); break;
    default: launch_tile<16>(g, L, scratch, counters, st); break;
  }
}

size_t split_doubles(const Gemm &g, const Launch &L) {
  return L.ksplit > 1 ? (size_t)L.ksplit * g.batch * (size_t)g.M * g.N : 0;
}

// First-use tuner. The model picks within a few per cent on most shapes but
// misses the better form on others (a sweep of the step's shapes: the best
// of single and pair forms 366 us against the model's 403 us for one core's
// products). So the first time a shape runs on a stream that is not being
// captured, the model's best single and pair candidates are timed (one
// warm-up and three launches each, on the call's own operands and output)
// and the fastest is kept for every later launch of the shape in the
// process -- also inside captured graphs. Candidates never need more split-K
// scratch than the model's plan, the size callers allocated; nothing is
// allocated; the stream is synchronized once per tuned shape. A shape first
// met inside a capture keeps the model's plan, and so do products under 1e7
// flops, products that accumulate into C, carry a skip flag, have
// device-side extents or whose C overlaps an operand, and every shape after
// the first 256 tuned in the process. Off by tt_gemm_autotune(0).
// Only for calls that keep their arithmetic (set_kept_arithmetic): the K split
// that is found here is the order of their sums.
std::atomic<bool> g_autotune{true};
constexpr double kTuneMinFlops = 1e7;    // smaller products keep the model's plan
constexpr int kTuneMaxShapes = 256;      // per process: bounds the tuning time
int g_tuned_shapes = 0;                  // guarded by g_exec_mu

// Elements spanned by an operand with the given strides (all non-negative).
long long span(const Gemm &g, long long s1, long long s2, long long sr, long long sc, int rows,
               int cols) {
  const long long b1max = (g.batch - 1) / g.bdiv, b2max = std::min(g.bdiv, g.batch) - 1;
  return b1max * s1 + b2max * s2 + (long long)(rows - 1) * sr + (long long)(cols - 1) * sc + 1;
}

// Products the tuner may run repeatedly with C as their output.
bool tunable(const Gemm &g) {
  if (g.beta != 0.0 || g.skip_dev != nullptr || g.dyn_dev != nullptr || g.C == nullptr) return false;
  if (g.sA1 < 0 || g.sA2 < 0 || g.sAm < 0 || g.sAk < 0 || g.sB1 < 0 || g.sB2 < 0 || g.sBk < 0 ||
      g.sBn < 0 || g.sC1 < 0 || g.sC2 < 0 || g.sCm < 0 || g.sCn < 0)
    return false;
  const char *c0 = reinterpret_cast<const char *>(g.C);
  const char *c1 = c0 + span(g, g.sC1, g.sC2, g.sCm, g.sCn, g.M, g.N) * (long long)sizeof(double);
  auto apart = [&](const double *x, long long n) {
    const char *x0 = reinterpret_cast<const char *>(x);
    const char *x1 = x0 + n * (long long)sizeof(double);
    return x == nullptr || x1 <= c0 || c1 <= x0;
  };
  return apart(g.A, span(g, g.sA1, g.sA2, g.sAm, g.sAk, g.M, g.K)) &&
         apart(g.B, span(g, g.sB1, g.sB2, g.sBk, g.sBn, g.K, g.N));
}

std::mutex g_exec_mu;
std::unordered_map<ShapeKey, Launch, ShapeHash> g_exec;

ShapeKey exec_key(const Gemm &g) {
  return {g.M, g.N, g.K, g.batch, g.bdiv, g.prec, g.sAk == 1 ? 1 : 0, g.sBn == 1 ? 1 : 0};
}

Launch tune(const Gemm &g, const Launch &Lm, double *scratch, int *counters, cudaStream_t st) {
  std::vector<std::pair<double, Launch>> cs, cp, pick;
  plan_candidates(g, false, cs);
  plan_candidates(g, true, cp);
  const size_t room = scratch ? split_doubles(g, Lm) : 0;
  auto ok = [&](const Launch &L) {
    return split_doubles(g, L) <= room && (L.ksplit == 1 || counters != nullptr);
  };
  for (auto *v : {&cs, &cp}) {
    std::sort(v->begin(), v->end(), [](const std::pair<double, Launch> &a,
                                       const std::pair<double, Launch> &b) { return a.first < b.first; });
    int taken = 0;
    for (const auto &x : *v) {
      if (taken == 6) break;
      if (!ok(x.second)) continue;
      pick.push_back(x);
      ++taken;
    }
  }
  if (pick.size() < 2) return Lm;
  // the candidates write C itself: every one computes the same product of
  // the same operands (exec_plan tunes only products with beta = 0, no skip
  // flag and C apart from A and B), and the chosen plan's launch follows
  Gemm gt = g;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  Launch best = Lm;
  float best_ms = 1e30f;
  bool fine = cudaEventCreate(&e0) == cudaSuccess && cudaEventCreate(&e1) == cudaSuccess;
  for (size_t i = 0; fine && i < pick.size(); ++i) {
    const Launch &L = pick[i].second;
    launch_plan(gt, L, scratch, counters, st);
    fine = cudaEventRecord(e0, st) == cudaSuccess;
    for (int r = 0; fine && r < 3; ++r) launch_plan(gt, L, scratch, counters, st);
    fine = fine && cudaEventRecord(e1, st) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess &&
           cudaGetLastError() == cudaSuccess;
    float ms = 0.0f;
    if (fine && cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess && ms < best_ms) {
      best_ms = ms;
      best = L;
    }
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaStreamSynchronize(st);
  cudaGetLastError();
  return fine ? best : Lm;
}

// HATT_GEMM_FORM=pair (read once): every FP64 shape takes the model's best
// paired tiling untimed -- a test hook that runs the paired kernel on every
// product of a workload.
bool force_pair() {
  static const bool v = [] {
    const char *e = getenv("HATT_GEMM_FORM");
    return e != nullptr && strcmp(e, "pair") == 0;
  }();
  return v;
}

// The plan a shape runs with: the tuned one once the shape has run (see tune).
Launch exec_plan(const Gemm &g, double *scratch, int *counters, cudaStream_t st) {
  const ShapeKey key = exec_key(g);
  {
    std::lock_guard<std::mutex> lock(g_exec_mu);
    const auto it = g_exec.find(key);
    if (it != g_exec.end()) return it->second;
  }
  Launch L = plan(g);
  if (force_pair() && g.prec == kPrecFP64) {
    std::vector<std::pair<double, Launch>> cp;
    plan_candidates(g, true, cp);
    const size_t room = scratch ? split_doubles(g, L) : 0;
    double best = 1e300;
    for (const auto &x : cp)
      if (x.first < best && split_doubles(g, x.second) <= room &&
          (x.second.ksplit == 1 || counters != nullptr)) {
        best = x.first;
        L = x.second;
      }
  }
  bool try_tune = !force_pair() && g_autotune.load(std::memory_order_relaxed) &&
                  g.prec == kPrecFP64 && 2.0 * g.M * g.N * (double)g.K * g.batch >= kTuneMinFlops &&
                  tunable(g);
  if (try_tune) {
    std::lock_guard<std::mutex> lock(g_exec_mu);
    try_tune = g_tuned_shapes < kTuneMaxShapes;
    if (try_tune) ++g_tuned_shapes;
  }
  if (try_tune) {
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusActive;
    if (cudaStreamIsCapturing(st, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone)
      L = tune(g, L, scratch, counters, st);
    cudaGetLastError();
  }
  std::lock_guard<std::mutex> lock(g_exec_mu);
  const auto it = g_exec.find(key);
  if (it != g_exec.end()) return it->second;   // another thread got there first
  if (g_exec.size() < (1u << 16)) g_exec.emplace(key, L);
  return L;
}

}  // namespace

void set_gemm_autotune(bool on) { g_autotune.store(on); }

namespace {
thread_local bool t_kept = false;

// Calls that keep their arithmetic, and, with HATT_GEMM_FORM=pair, all.
bool tiled_only() { return t_kept || force_pair(); }
}  // namespace
void set_kept_arithmetic(bool on) { t_kept = on; }
bool kept_arithmetic() { return t_kept; }

size_t gemm_scratch_doubles(const Gemm &g) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0) return 0;
  if (gemm_tc_supported(g)) return gemm_tc_scratch_doubles(g);
  if (!tiled_only()) {
    if (gemm_split_applicable(g)) return gemm_split_scratch_doubles(g);
    if (gemm_small_applicable(g)) return 0;
  }
  const Launch L = plan(g);
  return L.ksplit > 1 ? (size_t)L.ksplit * g.batch * (size_t)g.M * g.N : 0;
}

cudaError_t gemm_f64(const Gemm &g, double *scratch, cudaStream_t st) {
  if (g.M <= 0 || g.N <= 0 || g.batch <= 0) return cudaSuccess;
  if (g.K <= 0) {
    return cudaErrorInvalidValue;   // callers never issue empty contractions
  }
  if (gemm_tc_supported(g)) {                     // TF32 / BF16 operands: tensor cores
    const int slot = timer_begin(st);
    const cudaError_t e = gemm_tc(g, scratch, tile_counters(), st);
    timer_end(slot, st, 2.0 * g.M * g.N * (double)g.K * g.batch, g.role);
    return e;
  }
  const bool tiled = tiled_only();
  if (!tiled && gemm_split_applicable(g)) {       // digits on the FP16 tensor cores
    const int slot = timer_begin(st);
    const cudaError_t e = gemm_split(g, scratch, st);
    timer_end(slot, st, 2.0 * g.M * g.N * (double)g.K * g.batch, g.role);
    return e;
  }
  if (!tiled && gemm_small_applicable(g)) {
    const int slot = timer_begin(st);
    const cudaError_t e = gemm_small(g, st);
    timer_end(slot, st, 2.0 * g.M * g.N * (double)g.K * g.batch, g.role);
    return e;
  }
  int *counters = tile_counters();
  // a product with device-side extents is credited no flops: the host does
  // not know how many it does
  const double flops = g.dyn_dev ? 0.0 : 2.0 * g.M * g.N * (double)g.K * g.batch;
  Launch L = plan(g);
  if (L.ksplit > 1 && (scratch == nullptr || counters == nullptr)) return cudaErrorInvalidValue;
  if (tiled) L = exec_plan(g, scratch, counters, st);
  if (L.ksplit > 1 && (scratch == nullptr || counters == nullptr)) return cudaErrorInvalidValue;
  if ((long long)L.tiles_n * L.tiles_m * L.ksplit * g.batch >= (1LL << 31))
    return cudaErrorInvalidConfiguration;
  const int slot = timer_begin(st);
  launch_plan(g, L, scratch, counters, st);
  timer_end(slot, st, flops, g.role);
  return cudaGetLastError();
}

namespace {
thread_local int *t_tile_counters = nullptr;
}
void set_tile_counters(int *counters) { t_tile_counters = counters; }
int *tile_counters() { return t_tile_counters; }

}  // namespace hatt
