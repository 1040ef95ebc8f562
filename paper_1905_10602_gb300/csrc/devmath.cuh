// Device helpers shared by the kernels: FP64 <-> FP32 conversions on the integer
// pipes, warp reductions, the split cluster barrier.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "descs.h"

namespace ifmm {

// ---------------------------------------------------------------- FP64 <-> FP32 on the integer pipes
// GB300 executes double arithmetic and double<->float conversions on its narrow
// FP64 pipe (about 2 operations per clock per SM).  The FP32 kernels read and
// write FP64 storage, so they convert with integer operations on the IEEE-754
// fields instead, folding an optional power-of-two scale 2^sh into the
// exponent.  No path of either function uses a floating-point instruction (the
// compiler would evaluate a rare-path hardware conversion on every call and
// select).  d2f_pow2 rounds to nearest with ties away from zero (IEEE binary64
// -> binary32 keeps the top 23 of 52 fraction bits; the first dropped bit
// decides); results below the binary32 normal range become signed zero, above
// it infinity; infinity and NaN stay infinity and (quiet) NaN.  f2d_pow2 widens
// exactly (binary32 subnormals included); results below the binary64 normal
// range become signed zero, above it infinity.
__device__ __forceinline__ float d2f_pow2(double d, int sh) {
  const unsigned hi = (unsigned)__double2hiint(d), lo = (unsigned)__double2loint(d);
  const unsigned ah = hi & 0x7fffffffu, sg = hi & 0x80000000u;
  if (ah >= 0x7ff00000u) {
    const bool nan = ah > 0x7ff00000u || lo != 0u;
    return __uint_as_float(sg | 0x7f800000u | (nan ? 0x400000u | ((ah & 0x000fffffu) << 3) : 0u));
  }
  const int e = (int)(ah >> 20) + sh;  // biased binary64 exponent after scaling
  if (ah < 0x00100000u || e <= 896) return __uint_as_float(sg);
  if (e >= 1151) return __uint_as_float(sg | 0x7f800000u);
  unsigned f = ((unsigned)(e - 896) << 23) | ((ah & 0x000fffffu) << 3) | (lo >> 29);
  f += (lo >> 28) & 1u;  // a carry into the exponent is the correct rounding
  return __uint_as_float(sg | f);
}
__device__ __forceinline__ double f2d_pow2(float f, int sh) {
  const unsigned u = __float_as_uint(f);
  const unsigned a = u & 0x7fffffffu, sg = u & 0x80000000u;
  if (a == 0) return __hiloint2double((int)sg, 0);
  if (a >= 0x7f800000u) {
    const unsigned m = a & 0x007fffffu;  // NaN payload (0: infinity)
    return __hiloint2double((int)(sg | 0x7ff00000u | (m ? 0x80000u | (m >> 3) : 0u)), (int)(m << 29));
  }
  unsigned mant;
  int e;  // biased binary64 exponent
  if (a < 0x00800000u) {  // subnormal: a 2^-149, normalised
    const int lz = __clz((int)a) - 8;
    mant = (a << lz) & 0x007fffffu;
    e = 897 - lz + sh;
  } else {
    mant = a & 0x007fffffu;
    e = (int)(a >> 23) + 896 + sh;
  }
  if (e <= 0) return __hiloint2double((int)sg, 0);
  if (e >= 2047) return __hiloint2double((int)(sg | 0x7ff00000u), 0);
  return __hiloint2double((int)(sg | ((unsigned)e << 20) | (mant >> 3)), (int)(mant << 29));
}
// biased binary64 exponent of |d| (0 for zero and subnormals, 2047 for inf/NaN)
__device__ __forceinline__ int dexp(double d) { return (int)(((unsigned)__double2hiint(d) & 0x7fffffffu) >> 20); }

// d times 2^sh by its exponent field; results outside the normal range by ldexp
static __device__ __noinline__ double ldexp_rare(double d, int sh) { return ldexp(d, sh); }
__device__ __forceinline__ double scale_pow2(double d, int sh) {
  const int e = dexp(d);
  if (d == 0.0 || e == 2047) return d;
  if (e == 0 || e + sh <= 0 || e + sh >= 2047) return ldexp_rare(d, sh);
  return __hiloint2double(__double2hiint(d) + (sh << 20), __double2loint(d));
}
// value of a double as the arithmetic type TC, times 2^sh
template <typename TC>
__device__ __forceinline__ TC ld_tc(double d, int sh = 0) {
  if constexpr (sizeof(TC) == 4)
    return d2f_pow2(d, sh);
  else
    return sh ? ldexp(d, sh) : d;
}
// a TC value times 2^sh, as a double
template <typename TC>
__device__ __forceinline__ double st_tc(TC v, int sh = 0) {
  if constexpr (sizeof(TC) == 4)
    return f2d_pow2(v, sh);
  else
    return sh ? ldexp(v, sh) : v;
}

// ---------------------------------------------------------------- reductions
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename TC>
__device__ __forceinline__ TC warp_sum_t(TC v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// the warp's largest key (hi, lo), lexicographic, and the smallest index among
// the lanes that hold it; every lane gets the result
__device__ __forceinline__ void warp_max_key(unsigned& hi, unsigned& lo, int& i) {
  const unsigned mh = __reduce_max_sync(0xffffffffu, hi);
  const unsigned ml = __reduce_max_sync(0xffffffffu, hi == mh ? lo : 0u);
  i = (int)__reduce_min_sync(0xffffffffu, (hi == mh && lo == ml) ? (unsigned)i : 0x7fffffffu);
  hi = mh;
  lo = ml;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory"); }
// exponent shift that brings a block whose largest |entry| has biased binary64
// exponent emax into [0.5, 1) (0 for an all-zero block or one with inf/NaN)
__device__ __forceinline__ int pow2_shift(int emax) { return (emax <= 0 || emax >= 2047) ? 0 : 1022 - emax; }

// physical row of logical row i (QrcpDesc::rb, rs)
__device__ __forceinline__ long qr_row(const QrcpDesc& D, int i) {
  return D.rb > 0 ? (long)(i / D.rb) * D.rs + i % D.rb : (long)i;
}

}  // namespace ifmm
