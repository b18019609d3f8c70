// FP64 refinement of symmetric eigenvectors in one launch on a thread-block
// cluster (the eigen solves of the truncation sweep and of HPCRL-2's
// selection, for matrices up to kEigFusedMax): the Ogita-Aishima steps
// (Ogita & Aishima, JJIAM 2018) R = I - U^T U, S = U^T G U,
// l_i = s_ii / (1 - r_ii), E_ij = (s_ij + l_j r_ij) / (l_j - l_i) for
// separated pairs (rotations above 0.1 left out) and r_ij / 2 otherwise,
// U <- U (I + E), then Newton-Schulz steps E = R / 2, stopping after the
// first step whose correction is below 1e-9 -- the same steps and test as
// the launch-per-step path (four GEMM launches and one update launch per
// step, the later steps turned into no-ops by a device flag). Here one launch
// runs them all: CTA r of the cluster owns a slice of the columns of R, S and
// the new U, every CTA holds G and U whole in shared memory, slices and
// per-CTA norms travel through distributed shared memory (three cluster
// barriers per step), and the steps after convergence are not run at all.
// The FP32 start comes from the tridiagonal solver (k_trunc.cu) in U.
//
// FP64 arithmetic on GB300 runs on two lanes per SM: scalar FP64 work is done
// by one thread and broadcast through shared memory, never repeated by every
// thread. No spin-waits: hardware block and cluster barriers only, reached
// the same number of times by every CTA (the step count comes from values
// every CTA reads from the same shared words).
#include <cooperative_groups.h>
#include <algorithm>
#include <mutex>
#include "hatt_internal.cuh"

namespace cg = cooperative_groups;

namespace hatt {
namespace {

constexpr int kThreadsE = 512;
constexpr int kRefine = 3;          // Ogita-Aishima steps
constexpr int kOrth = 3;            // closing Newton-Schulz steps
constexpr double kStepConverged = 1e-9;
constexpr int kMaxCluster = 16;
constexpr int kColumnsMin = 8;      // least size of the whole-GPU form

// Block-wide sum / max of one double per thread. Only the warp shuffles run
// in every thread; the final combination of the per-warp values runs in
// thread 0 and is broadcast through shared memory: on GB300 every FP64
// instruction that all 512 threads execute costs the SM ~256 clocks.
__device__ __forceinline__ double blk_reduce(double v, double *red, bool is_max) {
  for (int o = 16; o > 0; o >>= 1) {
    const double x = __shfl_xor_sync(0xffffffffu, v, o);
    v = is_max ? fmax(v, x) : v + x;
  }
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  __syncthreads();
  if (l == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = red[0];
    for (int i = 1; i < (int)(blockDim.x >> 5); ++i) t = is_max ? fmax(t, red[i]) : t + red[i];
    red[32] = t;
  }
  __syncthreads();
  return red[32];
}


// U (c x c, row-major, device) holds the start on entry and the refined
// eigenvectors on return; *skip != 0 leaves it untouched.
__global__ void __launch_bounds__(kThreadsE, 1)
oa_cluster_kernel(const double *G, int c, double *Uout, double floor_norm, const int *skip) {
  pdl_enter();
  if (skip && *skip) return;           // every CTA reads the same word
  cg::cluster_group cl = cg::this_cluster();
  const int P = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int tid = threadIdx.x, nt = blockDim.x;
  const int w = (c + P - 1) / P;
  const int j0 = min(c, rank * w), j1 = min(c, j0 + w), wl = j1 - j0;
  extern __shared__ __align__(16) double sm[];
  double *Gs = sm;                     // c x c
  double *Us = Gs + c * c;             // c x c
  double *lam = Us + c * c;            // c
  double *part = lam + c;              // 3 x kMaxCluster
  double *work = part + 3 * kMaxCluster;
  double *Rs = work, *Ts = Rs + c * w, *Ss = Ts + c * w, *Ns = Ss + c * w;
  __shared__ double red[33];
  __shared__ double s_gn, s_delta, s_inv, s_stop;

  double g2 = 0.0;
  for (int e = tid; e < c * c; e += nt) {
    const double v = G[e];
    Gs[e] = v;
    Us[e] = Uout[e];
    g2 = fma(v, v, g2);
  }
  g2 = blk_reduce(g2, red, false);
  if (tid == 0) s_gn = sqrt(g2);
  cl.sync();                           // every CTA has started and loaded U
  const double u = 1.1102230246251565e-16;
  for (int it = 0; it < kRefine + kOrth; ++it) {
    const bool orth = it >= kRefine;
    // R = I - U^T U and T = G U on the own columns, then S = U^T T
    for (int e = tid; e < c * wl; e += nt) {
      const int i = e / wl, jj = e - i * wl, j = j0 + jj;
      double r = 0.0, t = 0.0;
      if (orth) {
        for (int k = 0; k < c; ++k) r = fma(Us[k * c + i], Us[k * c + j], r);
      } else {
        for (int k = 0; k < c; ++k) {
          const double ukj = Us[k * c + j];
          r = fma(Us[k * c + i], ukj, r);
          t = fma(Gs[i * c + k], ukj, t);
        }
      }
      Rs[i * w + jj] = ((i == j) ? 1.0 : 0.0) - r;
      Ts[i * w + jj] = t;
    }
    __syncthreads();
    if (!orth) {
      for (int e = tid; e < c * wl; e += nt) {
        const int i = e / wl, jj = e - i * wl;
        double s = 0.0;
        for (int k = 0; k < c; ++k) s = fma(Us[k * c + i], Ts[k * w + jj], s);
        Ss[i * w + jj] = s;
      }
      __syncthreads();
      for (int jj = tid; jj < wl; jj += nt) {      // l_j to every CTA
        const int j = j0 + jj;
        const double l = Ss[j * w + jj] / (1.0 - Rs[j * w + jj]);
        for (int q = 0; q < P; ++q) cl.map_shared_rank(lam, q)[j] = l;
      }
      double r2 = 0.0, s2 = 0.0;
      for (int e = tid; e < c * wl; e += nt) {
        const int i = e / wl, jj = e - i * wl, j = j0 + jj;
        const double r = Rs[i * w + jj];
        double sd = Ss[i * w + jj];
        if (i == j) sd -= Ss[j * w + jj] / (1.0 - Rs[j * w + jj]);
        r2 = fma(r, r, r2);
        s2 = fma(sd, sd, s2);
      }
      r2 = blk_reduce(r2, red, false);
      s2 = blk_reduce(s2, red, false);
      if (tid == 0)
        for (int q = 0; q < P; ++q) {
          double *pr = cl.map_shared_rank(part, q);
          pr[2 * rank] = r2;
          pr[2 * rank + 1] = s2;
        }
      cl.sync();
      if (tid == 0) {
        double R2 = 0.0, S2 = 0.0;
        for (int q = 0; q < P; ++q) {
          R2 += part[2 * q];
          S2 += part[2 * q + 1];
        }
        const double gn = s_gn;
        s_delta = fmax(2.0 * (sqrt(S2) + gn * sqrt(R2)),
                       64.0 * c * u * (floor_norm > 0.0 ? floor_norm : gn));
        s_inv = gn > 0.0 ? 1.0 / gn : 1.0;
      }
      __syncthreads();
    }
    const double delta = s_delta, inv = s_inv;
    // E (over R, in place), then the new columns U (I + E)
    double emax = 0.0;
    for (int e = tid; e < c * wl; e += nt) {
      const int i = e / wl, jj = e - i * wl, j = j0 + jj;
      const double r = Rs[i * w + jj];
      double E = 0.5 * r;
      if (!orth && i != j && fabs(lam[i] - lam[j]) > delta) {
        const float num = (float)(fma(lam[j], r, Ss[i * w + jj]) * inv);
        const float den = (float)((lam[j] - lam[i]) * inv);
        const float qv = __fdividef(num, den);
        if (fabsf(qv) <= 0.1f) E = (double)qv;
      }
      emax = fmax(emax, fabs(E));
      Rs[i * w + jj] = E;
    }
    __syncthreads();
    for (int e = tid; e < c * wl; e += nt) {
      const int i = e / wl, jj = e - i * wl, j = j0 + jj;
      double v = Us[i * c + j];
      for (int k = 0; k < c; ++k) v = fma(Us[i * c + k], Rs[k * w + jj], v);
      Ns[i * w + jj] = v;
    }
    emax = blk_reduce(emax, red, true);
    if (tid == 0)
      for (int q = 0; q < P; ++q) cl.map_shared_rank(part, q)[2 * kMaxCluster + rank] = emax;
    cl.sync();                         // every CTA has finished reading U
    for (int q = 0; q < P; ++q) {
      double *dst = cl.map_shared_rank(Us, q);
      for (int e = tid; e < c * wl; e += nt) {
        const int i = e / wl, jj = e - i * wl;
        dst[i * c + j0 + jj] = Ns[i * w + jj];
      }
    }
    cl.sync();
    if (tid == 0) {
      double mx = 0.0;
      for (int q = 0; q < P; ++q) mx = fmax(mx, part[2 * kMaxCluster + q]);
      s_stop = (mx <= kStepConverged) ? 1.0 : 0.0;
    }
    __syncthreads();
    if (s_stop != 0.0) break;          // the same decision in every CTA
  }
  for (int e = tid; e < c * wl; e += nt) {
    const int i = e / wl, jj = e - i * wl;
    Uout[i * c + j0 + jj] = Us[i * c + j0 + jj];
  }
}

// ------------------------------------------------------ whole-GPU form ---
// The same steps with one block per column in a cooperative launch: a step is
// 4 c^2 multiply-adds per block (R = U^T u and T = G u, S = U^T t, U E) and two grid
// barriers: after the eigenvalue estimates and the norms, and after the new
// columns, which travel through global memory. Used where the stream runs alone.
// Bound: below c ~ 64 the barriers (3000 to 4000 clocks each) and the dependent
// FP64 chains, above the FP64 unit of c SMs (the cluster form: of 16).
__device__ int g_refine_health = 0;    // kHealthTimeout: a barrier wait ran out
constexpr int kTG = 256;
constexpr int kMaxGroups = 8;
constexpr long long kBarrierCap = 1LL << 21;   // polls of one wait (seconds)

__device__ __forceinline__ bool column_barrier(int *bar, int target) {
  __syncthreads();
  int ok = 1;
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&bar[0], 1);
    volatile int *vb = bar;
    long long polls = 0;
    while (vb[0] < target) {
      if (vb[1] != 0) { ok = 0; break; }
      if (++polls > kBarrierCap) {
        atomicOr(&g_refine_health, kHealthTimeout);
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

__device__ __forceinline__ double warp_sum(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// U: start in, result out; Ub (c x c) and xch (6 c doubles) scratch; bar: two zero
// words.
__global__ void __launch_bounds__(kTG, 1)
refine_columns_kernel(const double *G, int c, double *U, double *Ub, double *xch, double floor_norm,
                      const int *skip, int *bar) {
  pdl_enter();
  if (skip && *skip) return;           // every block reads the same word
  extern __shared__ __align__(16) double sm[];
  const int ld = c | 1;                // odd: column and row walks without bank conflicts
  double *Gs = sm, *Us = Gs + c * ld;
  double *ru = Us + c * ld, *rt = ru + kMaxGroups * c;       // partial sums [group][i]
  double *uc = rt + kMaxGroups * c, *tc = uc + c, *rc = tc + c, *sc = rc + c, *lam = sc + c;
  double *lamg = xch, *normg = xch + c, *maxg = normg + 3 * c;
  __shared__ double s_gn, s_delta, s_inv, s_max[kTG / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int j = blockIdx.x, nb = gridDim.x;
  const int ng = min(kMaxGroups, kTG / c), q = tid / c, i = tid - q * c;
  const bool on = q < ng;
  for (int r = warp; r < c; r += kTG / 32)
    for (int l = lane; l < c; l += 32) {
      Gs[r * ld + l] = G[r * c + l];
      Us[r * ld + l] = U[r * c + l];
    }
  __syncthreads();
  const double u = 1.1102230246251565e-16;
  int target = 0;
  for (int it = 0; it < kRefine + kOrth; ++it) {
    const bool orth = it >= kRefine;
    double *dst = (it & 1) ? U : Ub;
    if (tid < c) uc[tid] = Us[tid * ld + j];
    __syncthreads();
    if (on) {                          // R = I - U^T U and T = G U, own column (G symmetric)
      double r0 = 0.0, r1 = 0.0, t0 = 0.0, t1 = 0.0;
      int k = q;
      for (; k + ng < c; k += 2 * ng) {
        const double x = uc[k], y = uc[k + ng];
        r0 = fma(Us[k * ld + i], x, r0);
        r1 = fma(Us[(k + ng) * ld + i], y, r1);
        if (!orth) {
          t0 = fma(Gs[k * ld + i], x, t0);
          t1 = fma(Gs[(k + ng) * ld + i], y, t1);
        }
      }
      if (k < c) {
        r0 = fma(Us[k * ld + i], uc[k], r0);
        if (!orth) t0 = fma(Gs[k * ld + i], uc[k], t0);
      }
      ru[q * c + i] = r0 + r1;
      rt[q * c + i] = t0 + t1;
    }
    __syncthreads();
    if (tid < c) {
      double r = ru[tid], t = rt[tid];
      for (int g = 1; g < ng; ++g) {
        r += ru[g * c + tid];
        if (!orth) t += rt[g * c + tid];
      }
      rc[tid] = (tid == j ? 1.0 : 0.0) - r;
      tc[tid] = t;
    }
    __syncthreads();
    if (!orth) {
      if (on) {                        // S = U^T T
        double s0 = 0.0, s1 = 0.0;
        int k = q;
        for (; k + ng < c; k += 2 * ng) {
          s0 = fma(Us[k * ld + i], tc[k], s0);
          s1 = fma(Us[(k + ng) * ld + i], tc[k + ng], s1);
        }
        if (k < c) s0 = fma(Us[k * ld + i], tc[k], s0);
        ru[q * c + i] = s0 + s1;
      }
      __syncthreads();
      if (tid < c) {
        double s = ru[tid];
        for (int g = 1; g < ng; ++g) s += ru[g * c + tid];
        sc[tid] = s;
      }
      __syncthreads();
      if (warp == 0) {                 // l_j and the column's shares of the norms
        const double l = sc[j] / (1.0 - rc[j]);
        double r2 = 0.0, s2 = 0.0, g2 = 0.0;
        for (int k = lane; k < c; k += 32) {
          const double sd = k == j ? sc[k] - l : sc[k], gv = Gs[k * ld + j];
          r2 = fma(rc[k], rc[k], r2);
          s2 = fma(sd, sd, s2);
          g2 = fma(gv, gv, g2);
        }
        r2 = warp_sum(r2);
        s2 = warp_sum(s2);
        g2 = warp_sum(g2);
        if (lane == 0) {
          lamg[j] = l;
          normg[3 * j] = r2;
          normg[3 * j + 1] = s2;
          normg[3 * j + 2] = g2;
        }
      }
      target += nb;
      if (!column_barrier(bar, target)) return;
      if (tid < c) lam[tid] = __ldcg(lamg + tid);
      if (warp == kTG / 32 - 1) {      // the same order in every block
        double r2 = 0.0, s2 = 0.0, g2 = 0.0;
        for (int k = lane; k < c; k += 32) {
          r2 += __ldcg(normg + 3 * k);
          s2 += __ldcg(normg + 3 * k + 1);
          g2 += __ldcg(normg + 3 * k + 2);
        }
        r2 = warp_sum(r2);
        s2 = warp_sum(s2);
        g2 = warp_sum(g2);
        if (lane == 0) {
          const double gn = sqrt(g2);
          s_delta = fmax(2.0 * (sqrt(s2) + gn * sqrt(r2)), 64.0 * c * u * (floor_norm > 0.0 ? floor_norm : gn));
          s_inv = gn > 0.0 ? 1.0 / gn : 1.0;
        }
      }
      __syncthreads();
    }
    double em = 0.0;                   // E (over R), then the new column U (I + E)
    if (tid < c) {
      const double r = rc[tid];
      double E = 0.5 * r;
      if (!orth && tid != j && fabs(lam[tid] - lam[j]) > s_delta) {
        const float num = (float)(fma(lam[j], r, sc[tid]) * s_inv);
        const float den = (float)((lam[j] - lam[tid]) * s_inv);
        const float qv = __fdividef(num, den);
        if (fabsf(qv) <= 0.1f) E = (double)qv;
      }
      em = fabs(E);
      rc[tid] = E;
    }
    for (int o = 16; o > 0; o >>= 1) em = fmax(em, __shfl_xor_sync(0xffffffffu, em, o));
    if (lane == 0) s_max[warp] = em;
    __syncthreads();
    if (on) {
      double s0 = 0.0, s1 = 0.0;
      int k = q;
      for (; k + ng < c; k += 2 * ng) {
        s0 = fma(Us[i * ld + k], rc[k], s0);
        s1 = fma(Us[i * ld + k + ng], rc[k + ng], s1);
      }
      if (k < c) s0 = fma(Us[i * ld + k], rc[k], s0);
      ru[q * c + i] = s0 + s1;
    }
    __syncthreads();
    if (tid < c) {
      double v = ru[tid];
      for (int g = 1; g < ng; ++g) v += ru[g * c + tid];
      v += uc[tid];
      uc[tid] = v;
      dst[tid * c + j] = v;
    }
    if (tid == 0) {
      double mx = s_max[0];
      for (int k = 1; k < kTG / 32; ++k) mx = fmax(mx, s_max[k]);
      maxg[(it & 1) * c + j] = mx;         // a closing step has one barrier: two buffers
    }
    target += nb;
    if (!column_barrier(bar, target)) return;
    double mx = 0.0;
    for (int k = lane; k < c; k += 32) mx = fmax(mx, __ldcg(maxg + (it & 1) * c + k));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (mx <= kStepConverged || it + 1 == kRefine + kOrth) {   // the same decision in every block
      // nobody reads U any more: every block has loaded the columns it needed
      if (dst != U && tid < c) U[tid * c + j] = uc[tid];
      return;
    }
    for (int r = warp; r < c; r += kTG / 32)
      for (int l = lane; l < c; l += 32) Us[r * ld + l] = __ldcg(dst + r * c + l);
    __syncthreads();
  }
}

size_t columns_smem(int c) {
  return ((size_t)2 * c * (c | 1) + (size_t)(2 * kMaxGroups + 5) * c) * sizeof(double);
}

int cluster_size_for(int c) { return c >= 32 ? 16 : (c >= 8 ? 8 : 1); }

size_t refine_smem(int c, int P) {
  const int w = (c + P - 1) / P;
  return ((size_t)2 * c * c + c + 3 * kMaxCluster + (size_t)4 * c * w) * sizeof(double);
}

}  // namespace

namespace {
// Largest cluster (16, else 8) the device can place with the kernel's shared
// memory, found once per device; 0 when not even 8 fit (then the caller keeps
// the launch-per-step path).
int g_max_cluster[kMaxDevices];
bool g_max_cluster_known[kMaxDevices];

std::mutex g_cluster_mu;

cudaError_t max_cluster(int *out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_cluster_mu);
  if (g_max_cluster_known[dev]) {
    *out = g_max_cluster[dev];
    return cudaSuccess;
  }
  e = cudaFuncSetAttribute(oa_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)refine_smem(kEigFusedMax, kMaxCluster));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(oa_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return e;
  int best = 0;
  for (int P : {kMaxCluster, 8}) {
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = P;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(P);
    cfg.blockDim = dim3(kThreadsE);
    cfg.dynamicSmemBytes = refine_smem(kEigFusedMax, P);
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int clusters = 0;
    if (cudaOccupancyMaxActiveClusters(&clusters, oa_cluster_kernel, &cfg) == cudaSuccess &&
        clusters > 0) {
      best = P;
      break;
    }
    cudaGetLastError();
  }
  g_max_cluster[dev] = best;
  g_max_cluster_known[dev] = true;
  *out = best;
  return cudaSuccess;
}
}  // namespace

cudaError_t refine_cluster_available(bool *ok) {
  int P = 0;
  const cudaError_t e = max_cluster(&P);
  *ok = (e == cudaSuccess && P > 0);
  return e;
}

cudaError_t refine_cluster(const double *G, int c, double *U, double floor_norm, const int *skip,
                           cudaStream_t st) {
  if (c < 1 || c > kEigFusedMax) return cudaErrorInvalidValue;
  int Pmax = 0;
  cudaError_t e = max_cluster(&Pmax);
  if (e != cudaSuccess) return e;
  if (Pmax == 0) return cudaErrorNotSupported;
  const int P = std::min(cluster_size_for(c), Pmax);
  const size_t smem = refine_smem(c, P);
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = P;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(P);
  cfg.blockDim = dim3(kThreadsE);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = programmatic_launch() ? 2 : 1;
  e = cudaLaunchKernelEx(&cfg, oa_cluster_kernel, G, c, U, floor_norm, skip);
  note_launch();
  return e;
}

cudaError_t refine_health_word(int *value, bool clear) {
  cudaError_t e = cudaMemcpyFromSymbol(value, g_refine_health, sizeof(int));
  if (e == cudaSuccess && clear && *value != 0) {
    const int zero = 0;
    e = cudaMemcpyToSymbol(g_refine_health, &zero, sizeof(int));
  }
  return e;
}

// Whether the whole-GPU form is taken: the stream runs alone, the device can
// place one block per column, and c has the scratch and the columns for it. It is
// the faster one at every size measured (us, this and the cluster form): c = 10 27
// and 34, 18 to 30 31 and 42, 34 51 and 69, 50 41 and 59, 90 79 and 215, 96 80 and 237.
cudaError_t refine_columns_available(int c, bool *ok) {
  *ok = false;
  if (c < kColumnsMin || c > kEigFusedMax || !programmatic_launch()) return cudaSuccess;
  int dev = 0, sms = 0, coop = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  *ok = e == cudaSuccess && coop != 0 && sms >= c;
  return e;
}

cudaError_t refine_columns(const double *G, int c, double *U, double *Ub, double *xch, double floor_norm,
                           const int *skip, int *bar, cudaStream_t st) {
  if (c < kColumnsMin || c > kEigFusedMax) return cudaErrorInvalidValue;
  cudaError_t e = cudaFuncSetAttribute(refine_columns_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)columns_smem(kEigFusedMax));
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(c);
  cfg.blockDim = dim3(kTG);
  cfg.dynamicSmemBytes = columns_smem(c);
  cfg.stream = st;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, refine_columns_kernel, G, c, U, Ub, xch, floor_norm, skip, bar);
  note_launch();
  return e;
}

}  // namespace hatt
