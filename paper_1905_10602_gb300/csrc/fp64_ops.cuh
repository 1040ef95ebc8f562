// Reciprocal and reciprocal square root in FP64 with few operations on GB300's
// narrow FP64 pipe: start values from the approximate units, moved between the
// formats by integer operations, then Newton steps.
#pragma once

#include <cuda_runtime.h>

namespace ifmm {

static __device__ __noinline__ double rsqrt_rare(double a) { return rsqrt(a); }
// 1/sqrt(a) to about an ulp: a = m 4^k, 1 <= m < 4; y0 = rsqrt(float(m)) 2^-k to
// ~2^-22, then one step y0 (1 + e/2 + 3 e^2 / 8), e = 1 - a y0^2 (the next term is
// below 2^-65).  Zero, subnormal, negative and non-finite arguments take CUDA's.
__device__ __forceinline__ double rsqrt_fp64(double a) {
  const int hi = __double2hiint(a);
  if ((unsigned)(hi - 0x00100000) >= 0x7fe00000u) return rsqrt_rare(a);
  const int k = ((hi >> 20) - 1023) >> 1;
  const unsigned f = __funnelshift_l((unsigned)__double2loint(a), (unsigned)(hi - (k << 21) - 0x38000000), 3);
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(__uint_as_float(f)));
  const unsigned u = __float_as_uint(y);
  const double y0 = __hiloint2double((int)(u >> 3) + 0x38000000 - (k << 20), (int)(u << 29));
  const double e = fma(-(a * y0), y0, 1.0);
  return fma(y0 * e, fma(0.375, e, 0.5), y0);
}

// 1/x: the approximate reciprocal refined by two Newton steps (its ~20 bits
// doubled twice); what it cannot take (subnormal or huge |x|) is divided
__device__ __forceinline__ double rcp_fp64(double x) {
  const unsigned e = ((unsigned)__double2hiint(x) >> 20) & 0x7ffu;
  if (e < 3u || e > 2042u) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  y = fma(fma(-x, y, 1.0), y, y);
  return fma(fma(-x, y, 1.0), y, y);
}
}  // namespace ifmm
