// The FP64 direct sums y = A x (Laplace and Helmholtz) with each unordered pair
// of points evaluated once: the kernels depend on |x_i - x_j| alone, so one
// value serves row i and row j.
//
// Bound: GB300's FP64 pipe (2 multiply-adds per clock and SM), so the FP64
// operations of a pair are what counts.  Everything else runs beside it: the
// start values of 1/r come from the FP32 reciprocal square root of the leading
// bits, moved between the formats by integer operations, and sine and cosine
// from a 64-entry table of one turn plus short Taylor sums.  13 FP64 operations
// per unordered pair (Laplace), 43 (Helmholtz).
//
// The points are cut into tiles of TB; a CTA takes a pair of tiles I <= J, each
// warp holding 32 targets of tile I and walking the sources of tile J in chunks
// of 32, lane l at source (l + step) mod 32, so that the lanes add to 32
// different column sums in the warp's shared memory without atomics.  Four steps
// are evaluated before their column sums are touched (independent FP64 chains).
// Row and column sums go to part[tile][point], written once each, which
// k_matvec64_sum adds in tile order: no result depends on scheduling.
//
// One product through bem_matvec, device vectors: n = 10,007 Laplace 8.49 ms ->
// 1.32 ms, n = 3,072 Helmholtz 10.7 ms -> 0.5 ms.  The full sums they
// replace had a thread per target and ceil(n / 256) CTAs.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fp64_ops.cuh"

namespace ifmm {

__device__ __noinline__ void sincos_rare(double a, double* s, double* c) { sincos(a, s, c); }

// sine and cosine of x: j = nearest integer to 32 x / pi, d = x - j pi / 32 in two
// steps (|d| <= pi / 64), table (cos, sin)(j pi / 32) and the Taylor sums of d to
// d^7 and d^8 (the next terms are below 2^-57).  |x| above 10^6 takes CUDA's.
__device__ __forceinline__ void sincos_fp64(double x, const double2* __restrict__ tab, double* sn, double* cs) {
  if ((__double2hiint(x) & 0x7fffffff) > 0x412e8480) {
    sincos_rare(x, sn, cs);
    return;
  }
  constexpr double kMagic = 6755399441055744.0;  // 1.5 * 2^52: the integer lands in the low word
  const double t = fma(x, 10.185916357881302, kMagic);
  const double2 T = tab[__double2loint(t) & 63];
  const double j = t - kMagic;
  // pi / 32 = hi + lo
  const double d = fma(-j, 3.827021247335479e-18, fma(-j, 0.09817477042468103, x));
  const double z = d * d;
  const double s = fma(fma(fma(z, -1.0 / 5040.0, 1.0 / 120.0), z, -1.0 / 6.0) * z, d, d);
  const double c = z * fma(fma(fma(z, 1.0 / 40320.0, -1.0 / 720.0), z, 1.0 / 24.0), z, -0.5);  // cos d - 1
  *sn = T.y + fma(T.x, s, T.y * c);
  *cs = T.x + fma(-T.y, s, T.x * c);
}

// (I, J), I <= J < T, of the tile pair b in row order
__device__ __forceinline__ void tile_pair(long b, int T, int* I_, int* J_) {
  int I = (int)((2.0 * T + 1.0 - sqrt((2.0 * T + 1.0) * (2.0 * T + 1.0) - 8.0 * (double)b)) / 2.0);
  auto first = [&](int i) { return (long)i * T - (long)i * (i - 1) / 2; };
  if (I < 0) I = 0;
  if (I > T - 1) I = T - 1;
  while (I > 0 && first(I) > b) --I;
  while (I < T - 1 && first(I + 1) <= b) ++I;
  *I_ = I;
  *J_ = I + (int)(b - first(I));
}

// CPLX: vectors of (re, im) pairs, part likewise (2 doubles per point)
template <int TB, bool CPLX>
__global__ void __launch_bounds__(TB) k_matvec64_sym(const double* __restrict__ px, const double* __restrict__ py,
                                                     const double* __restrict__ pz, const double* __restrict__ x,
                                                     double* __restrict__ part, int n, int T, double wk) {
  constexpr int DOF = CPLX ? 2 : 1, U = 4;
  __shared__ double sp[3][TB], sq[DOF][TB], col[TB / 32][DOF][TB];
  __shared__ double2 tab[CPLX ? 64 : 1];
  int I, J;
  tile_pair(blockIdx.x, T, &I, &J);
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int i = I * TB + tid, j = J * TB + tid;
  const bool live = i < n;
  double xi = 0, yi = 0, zi = 0, qi[DOF] = {};
  if (live) {
    xi = px[i];
    yi = py[i];
    zi = pz[i];
#pragma unroll
    for (int c = 0; c < DOF; ++c) qi[c] = x[(long)DOF * i + c];
  }
  sp[0][tid] = j < n ? px[j] : 0.0;
  sp[1][tid] = j < n ? py[j] : 0.0;
  sp[2][tid] = j < n ? pz[j] : 0.0;
#pragma unroll
  for (int c = 0; c < DOF; ++c) sq[c][tid] = j < n ? x[(long)DOF * j + c] : 0.0;
#pragma unroll
  for (int u = 0; u < TB / 32; ++u)
#pragma unroll
    for (int c = 0; c < DOF; ++c) col[u][c][tid] = 0.0;
  if (CPLX)
    for (int e = tid; e < 64; e += TB) {
      double s, c;
      sincospi(e / 32.0, &s, &c);
      tab[e] = make_double2(c, s);
    }
  __syncthreads();
  const int jn = n - J * TB;  // live sources of tile J
  double acc[DOF] = {};
  for (int c0 = 0; c0 < TB; c0 += 32) {
    for (int r = 0; r < 32; r += U) {
      double g[U][DOF];  // the kernel's value, real (and imaginary) part
      bool ok[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int s = c0 + ((lane + r + u) & 31);
        ok[u] = live && s < jn && (I != J || s != tid);
        const double dx = xi - sp[0][s], dy = yi - sp[1][s], dz = zi - sp[2][s];
        double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
        if (!ok[u]) r2 = 1.0;
        const double v = rsqrt_fp64(r2);
        if constexpr (CPLX) {
          double sn, cs;
          sincos_fp64(wk * (r2 * v), tab, &sn, &cs);
          g[u][0] = cs * v;
          g[u][1] = sn * v;
        } else {
          g[u][0] = v;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int s = c0 + ((lane + r + u) & 31);
        if (ok[u]) {
          if constexpr (CPLX) {
            acc[0] = fma(g[u][0], sq[0][s], fma(-g[u][1], sq[1][s], acc[0]));
            acc[1] = fma(g[u][1], sq[0][s], fma(g[u][0], sq[1][s], acc[1]));
          } else {
            acc[0] = fma(g[u][0], sq[0][s], acc[0]);
          }
          if (I != J) {  // a diagonal tile takes every ordered pair: rows only
            if constexpr (CPLX) {
              col[w][0][s] = fma(g[u][0], qi[0], fma(-g[u][1], qi[1], col[w][0][s]));
              col[w][1][s] = fma(g[u][1], qi[0], fma(g[u][0], qi[1], col[w][1][s]));
            } else {
              col[w][0][s] = fma(g[u][0], qi[0], col[w][0][s]);
            }
          }
        }
        __syncwarp();  // the next step's lanes add to these column sums
      }
    }
  }
  if (live)
#pragma unroll
    for (int c = 0; c < DOF; ++c) part[((long)J * n + i) * DOF + c] = acc[c];
  if (I != J) {
    __syncthreads();
    if (j < n)
#pragma unroll
      for (int c = 0; c < DOF; ++c) {
        double s = col[0][c][tid];
#pragma unroll
        for (int u = 1; u < TB / 32; ++u) s += col[u][c][tid];
        part[((long)I * n + j) * DOF + c] = s;
      }
  }
}

// y = diag x + scale * the tile sums, in tile order (dof entries per point)
__global__ void k_matvec64_sum(const double* __restrict__ part, int n, int T, const double* __restrict__ x,
                               double* __restrict__ y, double scale, double diag, double diag_im, int dof) {
  const long e = blockIdx.x * (long)blockDim.x + threadIdx.x, nd = (long)n * dof;
  if (e >= nd) return;
  double s = 0.0;
#pragma unroll 8
  for (int b = 0; b < T; ++b) s += part[b * nd + e];
  double d = diag * x[e];
  if (dof == 2) d = (e & 1) ? fma(diag_im, x[e - 1], d) : fma(-diag_im, x[e + 1], d);
  y[e] = fma(scale, s, d);
}

// Tile of the symmetric sums: 64 points while tiles of 128 would give fewer than
// eight tile pairs per SM (the last, partly filled wave then costs more than the
// smaller tile's extra column sums), else 128.
inline int matvec64_tile(int n) {
  const long t = ((long)n + 127) / 128;
  return t * (t + 1) / 2 < 8 * 152 ? 64 : 128;
}
// doubles of partial sums for n points, or 0 where they would exceed 8 GiB (the
// full sums k_matvec and k_matvec_c then have CTAs enough on their own)
inline size_t matvec64_part_doubles(int n, int dof) {
  const long tb = matvec64_tile(n), T = (n + tb - 1) / tb;
  const size_t d = (size_t)T * (size_t)n * dof;
  return d * sizeof(double) > ((size_t)8 << 30) ? 0 : d;
}

}  // namespace ifmm
