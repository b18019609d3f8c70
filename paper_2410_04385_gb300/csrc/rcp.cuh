// 1/x in FP64 for pivots in a bounded range (the Cholesky panels of k_qr.cu).
#pragma once

namespace hatt {

// x > 0 in [2^-100, 2^100): the range of the reciprocal below.
__device__ __forceinline__ bool rcp_range(double x) {
  return (unsigned)__double2hiint(x) - (923u << 20) < (200u << 20);
}
// 1/x for x in that range by one step of Householder's iteration of third order
// (A. S. Householder, The Numerical Treatment of a Single Nonlinear Equation, 1970)
// for f(r) = 1/r - x: r <- r (1 + e + e^2), e = 1 - x r, from an FP32 seed (rcp.approx
// of the truncated x, relative error below 2^-21). Three dependent FP64 multiply-adds
// leave e^3 < 2^-63 and one rounding. The conversions work on the bits: the FP64 unit
// takes ~100 clocks for each.
__device__ __forceinline__ double rcp_seeded(double x) {
  const unsigned xf = __funnelshift_l((unsigned)__double2loint(x), (unsigned)__double2hiint(x), 3) - (384u << 23);
  float f;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(f) : "f"(__uint_as_float(xf)));
  const unsigned u = __float_as_uint(f);
  double r = __hiloint2double((int)((u >> 3) + (896u << 20)), (int)(u << 29));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

}  // namespace hatt
