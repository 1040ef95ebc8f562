// Vector operations of GMRES: classical Gram-Schmidt applied twice, norms and
// linear combinations over the whole chip.
//
// Bound: memory (each pass reads the basis once) and, at the usual two to ten
// basis vectors, the launches.  A CTA owns a contiguous chunk of every vector
// and keeps its piece of w in shared memory; what it contributes to the dot
// products goes to part[vector][CTA], and the next kernel's CTAs each add those
// parts up in the same fixed order, so one Arnoldi step is four launches and one
// readback with no atomics and no result that depends on scheduling.  N =
// 65,536, eight iterations with a block-diagonal preconditioner: the vector work
// of the call 25 ms -> 0.3 ms (it was one CTA per operation, one warp for the
// updates).
#pragma once

#include <cuda_runtime.h>

namespace ifmm {

constexpr int kKryThreads = 256, kKryMaxChunk = 4096;

// sum over CTAs of part[0..nb) by one warp (every lane gets it)
__device__ __forceinline__ double kry_sum(const double* __restrict__ part, int nb, int lane) {
  double s = 0.0;
  for (int b = lane; b < nb; b += 32) s += part[b];
  return warp_sum(s);
}
// part[v nb + this CTA] = the chunk's share of V_v . w for v < nv (w's chunk in ws)
__device__ __forceinline__ void kry_dots(const double* __restrict__ V, long N, int nv, const double* ws, long e0,
                                         int cnt, double* __restrict__ part, int nb) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = kKryThreads / 32;
  for (int v = w; v < nv; v += nw) {
    const double* x = V + (long)v * N + e0;
    double s0 = 0.0, s1 = 0.0;
    int e = lane;
    for (; e + 32 < cnt; e += 64) {
      s0 = fma(x[e], ws[e], s0);
      s1 = fma(x[e + 32], ws[e + 32], s1);
    }
    if (e < cnt) s0 = fma(x[e], ws[e], s0);
    const double s = warp_sum(s0 + s1);
    if (lane == 0) part[(long)v * nb + blockIdx.x] = s;
  }
}

__global__ void __launch_bounds__(kKryThreads) k_kry_dots(const double* __restrict__ V, long N, int nv,
                                                          const double* __restrict__ w, int chunk,
                                                          double* __restrict__ part) {
  extern __shared__ double ksm[];
  const long e0 = (long)blockIdx.x * chunk;
  const int cnt = (int)min((long)chunk, N - e0);
  for (int e = threadIdx.x; e < cnt; e += kKryThreads) ksm[e] = w[e0 + e];
  __syncthreads();
  kry_dots(V, N, nv, ksm, e0, cnt, part, gridDim.x);
}

// h = the dot products in pin; w -= V h; pout = the parts of V . w (norm2 == 0)
// or of w . w (norm2 != 0) of the new w
__global__ void __launch_bounds__(kKryThreads) k_kry_update(const double* __restrict__ V, long N, int nv,
                                                            double* __restrict__ w, int chunk,
                                                            const double* __restrict__ pin, double* __restrict__ h,
                                                            double* __restrict__ pout, int norm2) {
  extern __shared__ double ksm[];
  double* hs = ksm + chunk;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nb = gridDim.x;
  for (int v = wp; v < nv; v += kKryThreads / 32) {
    const double s = kry_sum(pin + (long)v * nb, nb, lane);
    if (lane == 0) {
      hs[v] = s;
      if (blockIdx.x == 0) h[v] = s;
    }
  }
  __syncthreads();
  const long e0 = (long)blockIdx.x * chunk;
  const int cnt = (int)min((long)chunk, N - e0);
  for (int e = threadIdx.x; e < cnt; e += kKryThreads) {
    const double* x = V + e0 + e;
    double s = w[e0 + e];
#pragma unroll 4
    for (int v = 0; v < nv; ++v) s = fma(-hs[v], x[(long)v * N], s);
    w[e0 + e] = s;
    ksm[e] = s;
  }
  __syncthreads();
  if (norm2)
    kry_dots(w, N, 1, ksm, e0, cnt, pout, nb);
  else
    kry_dots(V, N, nv, ksm, e0, cnt, pout, nb);
}

// norm2 = the sum of the parts; v = w / sqrt(norm2) when that is positive
__global__ void __launch_bounds__(kKryThreads) k_kry_scale(const double* __restrict__ w, long N, int chunk,
                                                           const double* __restrict__ pin, double* __restrict__ norm2,
                                                           double* __restrict__ v) {
  const double s = kry_sum(pin, gridDim.x, threadIdx.x & 31);
  if (blockIdx.x == 0 && threadIdx.x == 0) *norm2 = s;
  const double nrm = sqrt(s);
  if (!(nrm > 0.0)) return;
  const double inv = 1.0 / nrm;
  const long e0 = (long)blockIdx.x * chunk;
  const int cnt = (int)min((long)chunk, N - e0);
  for (int e = threadIdx.x; e < cnt; e += kKryThreads) v[e0 + e] = inv * w[e0 + e];
}

// u = V y
__global__ void __launch_bounds__(kKryThreads) k_kry_combine(const double* __restrict__ V, long N, int nv,
                                                             const double* __restrict__ y, double* __restrict__ u) {
  const long e = blockIdx.x * (long)kKryThreads + threadIdx.x;
  if (e >= N) return;
  double s = 0.0;
#pragma unroll 4
  for (int v = 0; v < nv; ++v) s = fma(y[v], V[(long)v * N + e], s);
  u[e] = s;
}

__global__ void __launch_bounds__(kKryThreads) k_kry_add(const double* __restrict__ z, double* __restrict__ x, long N) {
  const long e = blockIdx.x * (long)kKryThreads + threadIdx.x;
  if (e < N) x[e] += z[e];
}

// r = b - r and the parts of r . r
__global__ void __launch_bounds__(kKryThreads) k_kry_residual(const double* __restrict__ b, double* __restrict__ r,
                                                              long N, int chunk, double* __restrict__ pout) {
  extern __shared__ double ksm[];
  const long e0 = (long)blockIdx.x * chunk;
  const int cnt = (int)min((long)chunk, N - e0);
  for (int e = threadIdx.x; e < cnt; e += kKryThreads) {
    const double s = b[e0 + e] - r[e0 + e];
    r[e0 + e] = s;
    ksm[e] = s;
  }
  __syncthreads();
  kry_dots(r, N, 1, ksm, e0, cnt, pout, gridDim.x);
}

}  // namespace ifmm
