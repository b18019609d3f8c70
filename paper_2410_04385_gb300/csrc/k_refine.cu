// FP64 refinement of symmetric eigenvectors in one launch (the eigen solves of the
// truncation sweep and of HPCRL-2's selection, for matrices up to kEigFusedMax):
// the Ogita-Aishima steps (Ogita & Aishima, JJIAM 2018) R = I - U^T U,
// S = U^T G U, l_i = s_ii / (1 - r_ii), E_ij = (s_ij + l_j r_ij) / (l_j - l_i) for
// separated pairs (rotations above 0.1 left out) and r_ij / 2 otherwise,
// U <- U (I + E), then Newton-Schulz steps E = R / 2, stopping after the
// first step whose correction is below 1e-9 -- the same steps and test as
// the launch-per-step path (four GEMM launches and one update launch per
// step, the later steps turned into no-ops by a device flag).
// The FP32 start comes from the tridiagonal solver (k_trunc.cu) in U.
//
// A column's products need only G, U and the column itself: a step is 4 c^2
// multiply-adds per column (R = U^T u and T = G u, S = U^T t, U E) and two
// barriers, after the eigenvalue estimates and norms and after the new columns,
// which travel through global memory. Two forms, bitwise the same:
//  * grid: one block per column in a cooperative launch, on calls whose stream
//    runs alone;
//  * cluster: up to 16 blocks of one cluster share the columns; stream lanes
//    (cooperative grids of several streams would run one after the other) and
//    c < 8.
// Bound: below c ~ 64 the barriers (3000 to 4000 clocks each in the grid form) and
// the dependent FP64 chains, above the FP64 unit of c SMs (cluster: of 16).
// Measured (us, grid and a cluster kernel): c = 10 27 and 34, 18 to 30 31 and 42,
// 34 51 and 69, 50 41 and 59, 90 79 and 215, 96 80 and 237.
#include <cooperative_groups.h>
#include <algorithm>
#include <mutex>
#include "hatt_internal.cuh"

namespace cg = cooperative_groups;

namespace hatt {
namespace {

constexpr int kRefine = 3;          // Ogita-Aishima steps
constexpr int kOrth = 3;            // closing Newton-Schulz steps
constexpr double kStepConverged = 1e-9;
constexpr int kMaxCluster = 16;
constexpr int kColumnsMin = 8;      // least size of the grid form

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
// words (grid form). Block b owns the columns b, b + nb, ...
template <bool CL>
__global__ void __launch_bounds__(kTG, 1)
refine_columns_kernel(const double *G, int c, double *U, double *Ub, double *xch, double floor_norm,
                      const int *skip, int *bar) {
  pdl_enter();
  if (skip && *skip) return;           // every block reads the same word
  extern __shared__ __align__(16) double sm[];
  const int ld = c | 1;                // odd: column and row walks without bank conflicts
  const int nb = gridDim.x, w = (c + nb - 1) / nb;
  double *Gs = sm, *Us = Gs + c * ld;
  double *ru = Us + c * ld, *rt = ru + kMaxGroups * c;       // partial sums [group][i]
  double *tc = rt + kMaxGroups * c, *lam = tc + c;
  double *ucs = lam + c, *rcs = ucs + w * c, *scs = rcs + w * c;   // per owned column
  double *lamg = xch, *normg = xch + c, *maxg = normg + 3 * c;
  __shared__ double s_delta, s_inv, s_max[kTG / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
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
  auto barrier = [&]() {
    if constexpr (CL) {
      asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
      return true;
    } else {
      target += nb;
      return column_barrier(bar, target);
    }
  };
  // sums of ru (and rt) over the groups, thread tid < c: entry tid
  auto over_groups = [&](const double *part) {
    double v = part[tid];
    for (int g = 1; g < ng; ++g) v += part[g * c + tid];
    return v;
  };
  for (int it = 0; it < kRefine + kOrth; ++it) {
    const bool orth = it >= kRefine;
    double *dst = (it & 1) ? U : Ub;
    for (int jj = 0, j = blockIdx.x; j < c; ++jj, j += nb) {
      double *uc = ucs + jj * c, *rc = rcs + jj * c, *sc = scs + jj * c;
      if (tid < c) uc[tid] = Us[tid * ld + j];
      __syncthreads();
      if (on) {                        // R = I - U^T U and T = G U, one column (G symmetric)
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
        rc[tid] = (tid == j ? 1.0 : 0.0) - over_groups(ru);
        if (!orth) tc[tid] = over_groups(rt);
      }
      __syncthreads();
      if (orth) continue;
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
      if (tid < c) sc[tid] = over_groups(ru);
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
    }
    if (!orth) {
      if (!barrier()) return;
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
    for (int jj = 0, j = blockIdx.x; j < c; ++jj, j += nb) {
      double *uc = ucs + jj * c, *rc = rcs + jj * c, *sc = scs + jj * c;
      double em = 0.0;                 // E (over R), then the new column U (I + E)
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
        const double v = over_groups(ru) + uc[tid];
        uc[tid] = v;
        dst[tid * c + j] = v;
      }
      if (tid == 0) {
        double mx = s_max[0];
        for (int k = 1; k < kTG / 32; ++k) mx = fmax(mx, s_max[k]);
        maxg[(it & 1) * c + j] = mx;   // a closing step has one barrier: two buffers
      }
      __syncthreads();
    }
    if (!barrier()) return;
    double mx = 0.0;
    for (int k = lane; k < c; k += 32) mx = fmax(mx, __ldcg(maxg + (it & 1) * c + k));
    for (int o = 16; o > 0; o >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (mx <= kStepConverged || it + 1 == kRefine + kOrth) {   // the same decision in every block
      // nobody reads U any more: every block has loaded what it needed of it
      if (dst != U && tid < c)
        for (int jj = 0, j = blockIdx.x; j < c; ++jj, j += nb) U[tid * c + j] = ucs[jj * c + tid];
      return;
    }
    for (int r = warp; r < c; r += kTG / 32)
      for (int l = lane; l < c; l += 32) Us[r * ld + l] = __ldcg(dst + r * c + l);
    __syncthreads();
  }
}

// The refinement of calls that keep their arithmetic (set_kept_arithmetic): CTA r
// of a cluster owns a slice of the columns of R, S and the new U, every CTA holds G
// and U whole in shared memory, and slices and per-CTA norms travel through
// distributed shared memory, three cluster barriers per step. Sums run over k in
// one chain, so the results differ from the kernel's above in the last bits.
// Bound by the FP64 units of its 16 SMs (c = 90: 215 us, above 79).
constexpr int kThreadsE = 512;

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
  double *part = lam + c;              // 4 x kMaxCluster
  double *work = part + 4 * kMaxCluster;
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
    // the CTAs' largest corrections: a closing step writes them before its first
    // barrier, while a slower CTA may still read those of the step before, so two
    // buffers (one value read twice would let the CTAs stop at different steps, with
    // writes to the shared memory of a CTA that has left)
    const int largest = (2 + (it & 1)) * kMaxCluster;
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
      for (int q = 0; q < P; ++q) cl.map_shared_rank(part, q)[largest + rank] = emax;
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
      for (int q = 0; q < P; ++q) mx = fmax(mx, part[largest + q]);
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

int cluster_size_for(int c) { return c >= 32 ? 16 : (c >= 8 ? 8 : 1); }

size_t refine_smem(int c, int P) {
  const int w = (c + P - 1) / P;
  return ((size_t)2 * c * c + c + 4 * kMaxCluster + (size_t)4 * c * w) * sizeof(double);
}

size_t columns_smem(int c, int blocks) {
  const int w = (c + blocks - 1) / blocks;
  return ((size_t)2 * c * (c | 1) + (size_t)(2 * kMaxGroups + 2 + 3 * w) * c) * sizeof(double);
}

// Largest cluster (16, else 8) the device can place with the kernels' shared
// memory, and its SMs if it launches cooperative grids, found once per device.
struct Device {
  bool known = false;
  int cluster = 0, kept_cluster = 0, coop_sms = 0;
};
Device g_device[kMaxDevices];
std::mutex g_device_mu;

cudaError_t device_info(Device *out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(g_device_mu);
  Device &D = g_device[dev];
  if (!D.known) {
    int sms = 0, coop = 0;
    e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(refine_columns_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)columns_smem(kEigFusedMax, 8));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(refine_columns_kernel<true>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(refine_columns_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)columns_smem(kEigFusedMax, kEigFusedMax));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(oa_cluster_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)refine_smem(kEigFusedMax, kMaxCluster));
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(oa_cluster_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    D.coop_sms = coop ? sms : 0;
    auto largest = [](auto kernel, int threads, size_t (*smem)(int, int)) {
      for (int P : {kMaxCluster, 8}) {
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = P;
        attr[0].val.clusterDim.y = 1;
        attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg = {};
        cfg.gridDim = dim3(P);
        cfg.blockDim = dim3(threads);
        cfg.dynamicSmemBytes = smem(kEigFusedMax, P);
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int clusters = 0;
        if (cudaOccupancyMaxActiveClusters(&clusters, kernel, &cfg) == cudaSuccess && clusters > 0) return P;
        cudaGetLastError();
      }
      return 0;
    };
    D.cluster = largest(refine_columns_kernel<true>, kTG, columns_smem);
    D.kept_cluster = largest(oa_cluster_kernel, kThreadsE, refine_smem);
    D.known = true;
  }
  *out = D;
  return cudaSuccess;
}

}  // namespace

cudaError_t refine_available(bool *ok) {
  Device D;
  const cudaError_t e = device_info(&D);
  *ok = e == cudaSuccess && (kept_arithmetic() ? D.kept_cluster : D.cluster) > 0;
  return e;
}

cudaError_t refine(const double *G, int c, double *U, double *Ub, double *xch, double floor_norm,
                   const int *skip, int *bar, cudaStream_t st) {
  if (c < 1 || c > kEigFusedMax) return cudaErrorInvalidValue;
  Device D;
  cudaError_t e = device_info(&D);
  if (e != cudaSuccess) return e;
  const bool kept = kept_arithmetic();
  if ((kept ? D.kept_cluster : D.cluster) == 0) return cudaErrorNotSupported;
  const bool grid = !kept && programmatic_launch() && c >= kColumnsMin && D.coop_sms >= c;
  const int blocks = grid ? c : std::min(cluster_size_for(c), kept ? D.kept_cluster : D.cluster);
  cudaLaunchAttribute attr[2];
  cudaLaunchConfig_t cfg = {};
  if (grid) {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.numAttrs = 1;
  } else {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.numAttrs = programmatic_launch() ? 2 : 1;
  }
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(kept ? kThreadsE : kTG);
  cfg.dynamicSmemBytes = kept ? refine_smem(c, blocks) : columns_smem(c, blocks);
  cfg.stream = st;
  cfg.attrs = attr;
  if (kept) {
    e = cudaLaunchKernelEx(&cfg, oa_cluster_kernel, G, c, U, floor_norm, skip);
    note_launch();
    return e;
  }
  e = cudaLaunchKernelEx(&cfg, grid ? refine_columns_kernel<false> : refine_columns_kernel<true>, G, c, U, Ub,
                         xch, floor_norm, skip, bar);
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

}  // namespace hatt
