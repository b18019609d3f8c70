// FP64 products too small to fill the device, C = alpha A B + beta C: every
// stage of a small recompression or inner product is a chain of them, each of
// which waits for the one before.
//
// Bound: latency (launch, one trip to L2, the dependent multiply-adds at ~65
// clocks), not arithmetic. So a block fetches its whole K at once (one exposure
// of the memory latency; the tiled kernel of k_gemm.cu pays it once per 16 to 80
// terms), K is split over the threads of the block and summed through shared
// memory (the tiled kernel splits it over blocks, with partial sums, a fence and
// an atomic in global memory), and a thread runs four sums side by side.
// Every sum has a fixed order.
// Measured in a chain (us, M x N x K; the tiled kernel in parentheses): 5 x 5 x 50
// 4.6 (6.2), 30 x 30 x 360 5.8 (10.7), 50 x 25 x 500 7.0 (12.4), 128 x 128 x 61 5.9
// (9.8), 64 x 64 x 500 9.0 (17.4), 34 x 34 x 34 4.5 (6.5), 8 x 8 x 8 3.8 (4.0).
#include <algorithm>
#include <cmath>
#include "hatt_internal.cuh"

namespace hatt {
namespace {

constexpr int kT = 256;
constexpr int kMaxGroups = 16;                 // K groups of a block
constexpr size_t kSmemMax = 110 * 1024;        // two blocks per SM
constexpr double kMaxFma = 3e6;

// rows x cols entries, cols with stride sf (the faster one in memory), rows with
// stride ss, to shared memory: entry (s, f) to dst[s ds + f df].
__device__ __forceinline__ void fetch(const double *p, long long sf, long long ss, int cols, int rows,
                                      double *dst, int df, int ds) {
  const int step_s = kT / cols, step_f = kT - step_s * cols;
  int s = (int)threadIdx.x / cols, f = (int)threadIdx.x - s * cols;
  while (s < rows) {
    const unsigned to = (unsigned)__cvta_generic_to_shared(dst + s * ds + f * df);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(to), "l"(p + s * ss + f * sf) : "memory");
    s += step_s;
    f += step_f;
    if (f >= cols) {
      f -= cols;
      ++s;
    }
  }
}

__global__ void __launch_bounds__(kT)
gemm_small_kernel(Gemm g, int bm, int bn, int tiles_n, int groups) {
  pdl_enter();
  if (g.skip_dev && *g.skip_dev) return;
  extern __shared__ double sm[];
  const int tid = threadIdx.x, K = g.K;
  const int tm = (int)(blockIdx.x / (unsigned)tiles_n), tn = (int)blockIdx.x - tm * tiles_n;
  const int b1 = (int)(blockIdx.y / (unsigned)g.bdiv), b2 = (int)blockIdx.y - b1 * g.bdiv;
  const int m0 = tm * bm, n0 = tn * bn, me = min(bm, g.M - m0), ne = min(bn, g.N - n0);
  double *As = sm, *Bs = As + (size_t)bm * K, *red = Bs + (size_t)bn * K;     // [k][m], [k][n], [group][out]
  const double *A = g.A + b1 * g.sA1 + b2 * g.sA2 + m0 * g.sAm;
  const double *B = g.B + b1 * g.sB1 + b2 * g.sB2 + n0 * g.sBn;
  if (g.sAk == 1) fetch(A, 1, g.sAm, K, me, As, bm, 1);
  else fetch(A, g.sAm, g.sAk, me, K, As, 1, bm);
  if (g.sBn == 1) fetch(B, 1, g.sBk, ne, K, Bs, 1, bn);
  else fetch(B, g.sBk, g.sBn, K, ne, Bs, bn, 1);
  const double alpha = g.alpha * (g.alpha_dev ? *g.alpha_dev : 1.0);
  const int outs = bm * bn;
  const int q = tid / outs, o = tid - q * outs, m = o / bn, n = o - m * bn;
  const bool mine = q < groups && m < me && n < ne;
  double *c = g.C + b1 * g.sC1 + b2 * g.sC2 + (m0 + m) * g.sCm + (n0 + n) * g.sCn;
  const double old = mine && q == 0 && g.beta != 0.0 ? *c : 0.0;
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  double acc = 0.0;
  if (mine) {
    double a1 = 0.0, a2 = 0.0, a3 = 0.0;
    const double *a = As + m, *b = Bs + n;
    const int sa = groups * bm, sb = groups * bn;
    a += q * bm;
    b += q * bn;
    int k = q;
    for (; k + 3 * groups < K; k += 4 * groups) {
      acc = fma(a[0], b[0], acc);
      a1 = fma(a[sa], b[sb], a1);
      a2 = fma(a[2 * sa], b[2 * sb], a2);
      a3 = fma(a[3 * sa], b[3 * sb], a3);
      a += 4 * sa;
      b += 4 * sb;
    }
    for (; k < K; k += groups) {
      acc = fma(*a, *b, acc);
      a += sa;
      b += sb;
    }
    if (K > 3 * groups) acc = (acc + a1) + (a2 + a3);
  }
  if (groups > 1) {
    if (mine && q > 0) red[q * outs + o] = acc;
    __syncthreads();
    if (!mine || q > 0) return;
    double r = 0.0;
    int i = 1;
    for (; i + 1 < groups; i += 2) {
      acc += red[i * outs + o];
      r += red[(i + 1) * outs + o];
    }
    if (i < groups) acc += red[i * outs + o];
    acc += r;
  }
  if (mine) {
    const double v = alpha * acc;
    *c = g.beta != 0.0 ? fma(g.beta, old, v) : v;
  }
}

struct Tile {
  int bm = 0, bn = 0, groups = 0;          // bm = 0: not taken
};

size_t small_smem(const Tile &t, int K) {
  return ((size_t)(t.bm + t.bn) * K + (t.groups > 1 ? (size_t)t.groups * t.bm * t.bn : 0)) * sizeof(double);
}

// Predicted clocks of the product after its launch: the fetch (latency, then 12
// clocks per warp of 8-byte copies), the multiply-adds (a chain of ~65 clocks each
// for a warp; 16 clocks per warp on the SM's FP64 unit, shared by its blocks)
// and the sum over the groups.
double tile_clocks(const Gemm &g, const Tile &t, int sms) {
  const double outs = (double)t.bm * t.bn;
  const double blocks = (double)((g.M + t.bm - 1) / t.bm) * ((g.N + t.bn - 1) / t.bn) * g.batch;
  const double per_sm = std::ceil(blocks / sms);
  const double steps = std::ceil((double)g.K / t.groups);
  const double issue = 16.0 * std::ceil(outs * t.groups / 32.0) * steps;
  const double chain = 65.0 * std::ceil(steps / 4.0);
  const double copies = 12.0 * std::ceil((double)(t.bm + t.bn) * g.K / 32.0);
  const double resident = std::min(per_sm, std::max(1.0, std::floor(220.0 * 1024.0 / (double)(small_smem(t, g.K) + 1024))));
  return 900.0 * std::ceil(per_sm / resident) + per_sm * copies + std::max(chain, per_sm * issue) +
         (t.groups > 1 ? 100.0 + 33.0 * t.groups : 0.0);
}

Tile choose_tile(const Gemm &g, int sms) {
  static const int edges[] = {1, 2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 25, 32, 48, 64, 128, 256};
  Tile best;
  double best_t = 1e30;
  for (int em : edges) {
    const int bm = std::min(em, g.M);
    for (int en : edges) {
      const int bn = std::min(en, g.N);
      if (bm * bn > kT) break;
      Tile t;
      t.bm = bm;
      t.bn = bn;
      t.groups = std::max(1, std::min({kMaxGroups, kT / (bm * bn), (g.K + 3) / 4}));
      if (small_smem(t, g.K) <= kSmemMax) {
        const double c = tile_clocks(g, t, sms);
        if (c < best_t) {
          best_t = c;
          best = t;
        }
      }
      if (bn == g.N) break;
    }
    if (bm == g.M) break;
  }
  return best;
}

// The choice for the sizes of g; the last ones are remembered per thread (a
// pure function of the sizes).
Tile tile_for(const Gemm &g) {
  struct Entry {
    int M = 0, N = 0, K = 0, batch = 0;
    Tile t;
  };
  thread_local Entry cache[256];
  const unsigned h = ((unsigned)g.M * 0x9E3779B1u) ^ ((unsigned)g.N * 0x85EBCA77u) ^
                     ((unsigned)g.K * 0xC2B2AE3Du) ^ ((unsigned)g.batch * 0x27D4EB2Fu);
  Entry &e = cache[(h >> 16) & 255];
  if (e.M != g.M || e.N != g.N || e.K != g.K || e.batch != g.batch) {
    e.M = g.M;
    e.N = g.N;
    e.K = g.K;
    e.batch = g.batch;
    e.t = choose_tile(g, 152);
  }
  return e.t;
}

}  // namespace

// FP64 products of at most kMaxFma multiply-adds with fixed extents. From there
// on the tiled kernel's larger tiles fetch less (us, this and the tiled kernel):
// 200 x 200 x 50 (2 M) 8.6 and 11.3, 50 x 50 x 1280 (3.2 M) 17.9 and 17.7, 32
// products 50 x 50 x 50 (4 M) 17.7 and 17.1, 400 products 18 x 30 x 18 (3.9 M) 15.8
// and 14.0.
bool gemm_small_applicable(const Gemm &g) {
  if (g.prec != kPrecFP64 || g.dyn_dev != nullptr || g.batch > 65535) return false;
  if ((double)g.M * g.N * (double)g.K * g.batch > kMaxFma) return false;
  const Tile t = tile_for(g);
  return t.bm > 0 &&
         (long long)((g.M + t.bm - 1) / t.bm) * ((g.N + t.bn - 1) / t.bn) < (1LL << 31);
}

cudaError_t gemm_small(const Gemm &g, cudaStream_t st) {
  const Tile t = tile_for(g);
  const int tiles_n = (g.N + t.bn - 1) / t.bn, tiles_m = (g.M + t.bm - 1) / t.bm;
  const size_t smem = small_smem(t, g.K);
  if (smem > 48 * 1024) {
    const cudaError_t e =
        cudaFuncSetAttribute(gemm_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
    if (e != cudaSuccess) return e;
  }
  launch_k(gemm_small_kernel, dim3((unsigned)(tiles_n * tiles_m), (unsigned)g.batch), kT, smem, st, g, t.bm,
           t.bn, tiles_n, t.groups);
  note_launch();
  return cudaGetLastError();
}

}  // namespace hatt
