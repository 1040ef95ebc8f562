// The explicit inverse of one large FP64 matrix (the level-1 system): blocked
// in-place Gauss-Jordan with partial pivoting, its rank-32 updates on the tensor
// cores as products of 8-bit digits.
//
// A panel of nb = 32 columns K is exchanged on its own, rows spread over the CTAs
// of one cluster; with P its pivot rows, B = A(P, K) and A' the exchanged panel
// (A'(P, K) = B^-1, A'(i, K) = -A(i, K) B^-1), every other column is
//   A(i, J) += A'(i, K) A(P, J)   with the rows P of A(., J) taken as zero,
// one product per panel.  Rows are never moved: after the last panel row p_k holds
// x_k, so Ainv(k, p_k') = M(p_k, k') is written out at the end.
//
// The product splits its operands into digits (the error-free splitting of Ozaki,
// Ogita, Oishi and Rump): each row of A' and each column of A(P, J) is scaled by a
// power of two to |m| < 1 and rounded to seven signed 8-bit digits, 55 bits below
// that power; products of digits summed over 32 terms and up to seven digit pairs
// stay below 2^22, so the FP32 accumulators are exact integers, and the eight
// orders i + j <= 7 are added up in 64-bit integers.  With r and c the largest
// entries of a row of A' and a column of A(P, J), the operands' rounding leaves
// 32 * 2^-54 r c over the 32 terms at most and the dropped orders 2^-54.7 r c: the
// error is relative to r c, not to the terms, and an entry 2^-k below its row's or
// column's largest keeps 55 - k bits.  Rows of very different size would put the
// large entries of A' against the small ones of A(P, J) (A' is graded by 1/d_p, A(P, J)
// by d_p), so column p of A' is taken times 2^s_p and row p of A(P, J) times 2^-s_p, s_p
// the exponent of the largest entry of row p of the matrix: what a power-of-two
// scaling of the rows would give, with the pivots of the unscaled matrix.  (The
// columns' sizes cancel without it.)  Half the rows times 2^-40, n = 200, emulated in
// NumPy: error 3.8e10 u |X||A||X| without, 0.4 u with, 0.5 u in plain FP64 elimination.
// 34 MMA passes replace the FP64 multiply-adds, whose pipe (2 per clock and SM)
// bounds the plain elimination: n = 3,628 needs 90 ms there.  What bounds it now is
// the panels' chain of n pivot steps (one cluster barrier each).  The two launches
// per column it replaces: n = 3,628 243 -> 52 ms, n = 2,296 69 -> 18, n = 1,417 29 -> 7.9.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "devmath.cuh"
#include "fp64_ops.cuh"

namespace ifmm {

constexpr int kBiNb = 32;       // panel width
constexpr int kBiSlices = 7;    // 8-bit digits per entry
constexpr int kBiTile = 64;     // output tile of the product
constexpr int kBiPitch = 40;    // shared-memory row of digits: 32 + 8 (80 bytes: ldmatrix free of bank conflicts)
constexpr int kBiThreads = 512;
constexpr int kBiBad = 1 << 20; // exponent of a row or column with an infinity or NaN

// panel rows in one CTA (two per thread at most)
inline int bi_rows(int n, int R) { return (n + R - 1) / R; }
inline size_t bi_panel_bytes(int n, int R) {
  return (size_t)bi_rows(n, R) * (kBiNb + 1) * sizeof(double) + (size_t)2 * R * (kBiNb + 2) * sizeof(double);
}
// device scratch: digits of A' and of the pivot rows (n x 32 each and slice), their exponents, the rows' scales, the
// used rows
inline size_t bi_work_bytes(int n) {
  const size_t np = ((size_t)n + kBiTile - 1) / kBiTile * kBiTile;
  return 2 * kBiSlices * np * kBiNb * 2 + 3 * np * sizeof(int) + np + 1024;
}
struct BiWork {
  uint16_t *da, *db;  // digits [slice][row or column][32], bfloat16
  int *ea, *eb;       // exponents
  int* es;            // biased exponent of the largest entry of each row of the matrix
  unsigned char* used;
  int np;             // rows and columns, padded to the tile
};

constexpr int kBiNone = -0x100000;  // no nonzero entry

// The power of two that row p counts as (its largest entry's; an infinity or NaN, or
// nothing but zeros and subnormals: 1)
__device__ __forceinline__ int bi_scale(const BiWork& w, int p) {
  const int e = w.es[p];
  return e > 0 && e < 2047 ? e - 1023 : 0;
}
// es (zeroed) = the rows' largest biased exponents; a thread per row, 64 columns a CTA
__global__ void __launch_bounds__(256) k_bi_scales(const double* __restrict__ A, int n, BiWork w) {
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= n) return;
  const int j1 = min(n, (int)(blockIdx.y + 1) * 64);
  int e = 0;
  for (int j = blockIdx.y * 64; j < j1; ++j) e = max(e, dexp(A[i + (long)j * n]));
  atomicMax(w.es + i, e);
}

// The seven digits of x / 2^e (|x| < 2^e) as bfloat16 bits: d[s] has weight
// 2^(-7 - 8 s); rounded to 55 bits.
__device__ __forceinline__ void bi_digits(double x, int e, unsigned (&d)[kBiSlices]) {
  const int ex = dexp(x);
  long long M = 0;
  const int sh = e + 1023 - 1 - ex;  // >= 0: how far x's leading bit lies below 2^(e-1)
  if (ex > 0 && sh < 57) {
    const long long mant =
        ((long long)(__double2hiint(x) & 0xfffff) << 32 | (unsigned)__double2loint(x)) | (1ll << 52);
    M = sh <= 2 ? mant << (2 - sh) : (mant + (1ll << (sh - 3))) >> (sh - 2);
    if (__double2hiint(x) < 0) M = -M;
  }
#pragma unroll
  for (int s = kBiSlices - 1; s >= 0; --s) {
    const int q = s ? (int)(signed char)(M & 0xff) : (int)M;
    M = (M - q) >> 8;
    // |q| <= 128: exact in bfloat16 (the float through the 1.5 * 2^23 trick)
    d[s] = __float_as_uint(__int_as_float(0x4B400000 + q) - 12582912.f) >> 16;
  }
}

// Columns k0 .. k0 + kb of A exchanged, one cluster; piv, used and A' digits out.
__global__ void __launch_bounds__(kBiThreads) k_bi_panel(double* __restrict__ A, int n, int k0, int kb,
                                                         int* __restrict__ piv, BiWork w, int* __restrict__ info) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int R = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  if (info[0] != 0) return;  // the same for every CTA: written by an earlier launch only
  const int chunk = (n + R - 1) / R, r0 = min(n, rank * chunk), ml = min(n, r0 + chunk) - r0;
  extern __shared__ __align__(16) double bsm[];
  double* P = bsm;                            // [32][chunk]
  double* cb = P + (size_t)kBiNb * chunk;     // column k before the step
  double* rowb = cb + chunk;                  // [2][R][32]: the CTAs' candidate rows, scaled
  unsigned long long* kv = (unsigned long long*)(rowb + 2 * R * kBiNb);  // [2][R] keys
  int* ki = (int*)(kv + 2 * R);               // [2][R] rows
  __shared__ unsigned rh[16], rl[16];
  __shared__ int ri[16];
  __shared__ int sx[kBiNb];  // the panel's pivot rows, then their scales
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  for (int c = wp; c < kBiNb; c += kBiThreads / 32)
    for (int i = lane; i < ml; i += 32) P[(size_t)c * chunk + i] = c < kb ? A[(r0 + i) + (long)(k0 + c) * n] : 0.0;
  bool used[2];
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int i = tid + v * kBiThreads;
    used[v] = i >= ml || w.used[r0 + (i < ml ? i : 0)] != 0;
  }
  cl.sync();
  int bad = 0;
  for (int k = 0; k < kb; ++k) {
    const int b = k & 1;
    // this CTA's candidate: largest |P(i, k)| of its unused rows, ties to the smallest row
    unsigned hi = 0, lo = 0;
    int bi = 0x7fffffff;
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int i = tid + v * kBiThreads;
      if (i >= ml) continue;
      const double x = P[(size_t)k * chunk + i];
      cb[i] = x;
      const unsigned h = (unsigned)__double2hiint(x) & 0x7fffffffu, l = (unsigned)__double2loint(x);
      const bool nan = h > 0x7ff00000u || (h == 0x7ff00000u && l);
      if (!used[v] && !nan && (bi == 0x7fffffff || h > hi || (h == hi && l > lo))) {
        hi = h;
        lo = l;
        bi = i;
      }
    }
    warp_max_key(hi, lo, bi);
    if (lane == 0) {
      rh[wp] = hi;
      rl[wp] = lo;
      ri[wp] = bi;
    }
    __syncthreads();
    if (wp == 0) {
      hi = lane < 16 ? rh[lane] : 0u;
      lo = lane < 16 ? rl[lane] : 0u;
      bi = lane < 16 ? ri[lane] : 0x7fffffff;
      warp_max_key(hi, lo, bi);
      // lane c: entry c of the candidate row, scaled by the reciprocal pivot
      const bool ok = (hi | lo) != 0;
      const double x = ok ? P[(size_t)lane * chunk + bi] : 0.0;
      const double q = rcp_fp64(ok ? __shfl_sync(0xffffffffu, x, k) : 1.0);
      const double r = lane == k ? q : x * q;
      for (int t = 0; t < R; ++t) cl.map_shared_rank(rowb, t)[(b * R + rank) * kBiNb + lane] = r;
      if (lane < R) {
        cl.map_shared_rank(kv, lane)[b * R + rank] = (unsigned long long)hi << 32 | lo;
        cl.map_shared_rank(ki, lane)[b * R + rank] = ok ? r0 + bi : 0x7fffffff;
      }
    }
    cl.sync();
    const unsigned long long kk = lane < R ? kv[b * R + lane] : 0ull;
    hi = (unsigned)(kk >> 32);
    lo = (unsigned)kk;
    int p = lane < R ? ki[b * R + lane] : 0x7fffffff;
    warp_max_key(hi, lo, p);
    if ((hi | lo) == 0) {
      bad = k0 + k + 1;
      break;
    }
    if (tid == 0) {
      sx[k] = p;
      if (rank == 0) piv[k0 + k] = p;
    }
    const double* row = rowb + (b * R + p / chunk) * kBiNb;
    const int pl = p - r0;  // the pivot's local row, if it is here
#pragma unroll
    for (int v = 0; v < 2; ++v) used[v] = used[v] || tid + v * kBiThreads == pl;
    // (32 rows, 4 columns) items over the warps
    const int nrb = (ml + 31) >> 5;
    for (int e = wp; e < nrb * (kBiNb / 4); e += kBiThreads / 32) {
      const int rb = e >> 3, c0 = (e & 7) * 4, i = rb * 32 + lane;
      if (i >= ml) continue;
      const double ci = -cb[i];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int c = c0 + u;
        const double r = row[c];
        double* a = P + (size_t)c * chunk + i;
        *a = i == pl ? r : (c == k ? ci * r : fma(ci, r, *a));
      }
    }
    __syncthreads();
  }
  if (bad) {
    if (rank == 0 && tid == 0) info[0] = bad;
    cl.sync();
    return;
  }
  if (tid < kBiNb) sx[tid] = tid < kb ? bi_scale(w, sx[tid]) : 0;
  __syncthreads();
  for (int c = wp; c < kb; c += kBiThreads / 32)
    for (int i = lane; i < ml; i += 32) A[(r0 + i) + (long)(k0 + c) * n] = P[(size_t)c * chunk + i];
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const int i = tid + v * kBiThreads;
    if (i >= ml) continue;
    w.used[r0 + i] = used[v];
    // digits of row r0 + i, entry c times 2^sx[c]
    int e = kBiNone;
    bool fin = true;
    for (int c = 0; c < kBiNb; ++c) {
      const int ex = dexp(P[(size_t)c * chunk + i]);
      fin = fin && ex < 2047;
      if (ex > 0) e = max(e, ex + sx[c]);
    }
    if (e == kBiNone) e = 0;
    w.ea[r0 + i] = fin ? e - 1022 : kBiBad;
    for (int c0 = 0; c0 < kBiNb; c0 += 8) {
      unsigned lo16[kBiSlices][4];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        unsigned d[kBiSlices];
        bi_digits(fin ? P[(size_t)(c0 + u) * chunk + i] : 0.0, e - 1022 - sx[c0 + u], d);
#pragma unroll
        for (int s = 0; s < kBiSlices; ++s) lo16[s][u >> 1] = (u & 1) ? lo16[s][u >> 1] | d[s] << 16 : d[s];
      }
#pragma unroll
      for (int s = 0; s < kBiSlices; ++s)
        *(uint4*)(w.da + ((size_t)s * w.np + r0 + i) * kBiNb + c0) =
            make_uint4(lo16[s][0], lo16[s][1], lo16[s][2], lo16[s][3]);
    }
  }
  cl.sync();
}

// Digits of the pivot rows of panel k0 in every other column (a warp per column,
// lane s: row p = piv[k0 + s], times 2^-s_p), which are then zero; the panel's own columns get zero
// digits (their product must add nothing).
__global__ void __launch_bounds__(256) k_bi_rows(double* __restrict__ A, int n, int k0, int kb,
                                                 const int* __restrict__ piv, BiWork w, const int* __restrict__ info) {
  if (info[0] != 0) return;
  const int j = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (j >= w.np) return;
  const bool own = j >= n || (j >= k0 && j < k0 + kb);
  double x = 0.0;
  int sc = 0;
  if (!own && lane < kb) {
    const int p = piv[k0 + lane];
    double* a = A + p + (long)j * n;
    sc = bi_scale(w, p);
    x = *a;
    *a = 0.0;
  }
  const int ex = dexp(x);
  const bool fin = __all_sync(0xffffffffu, ex < 2047);
  int e = __reduce_max_sync(0xffffffffu, ex > 0 ? ex - sc : kBiNone);
  if (e == kBiNone) e = 0;
  if (lane == 0) w.eb[j] = fin ? e - 1022 : kBiBad;
  unsigned d[kBiSlices];
  bi_digits(fin ? x : 0.0, e - 1022 + sc, d);
#pragma unroll
  for (int s = 0; s < kBiSlices; ++s) w.db[((size_t)s * w.np + j) * kBiNb + lane] = (uint16_t)d[s];
}

__device__ __forceinline__ void ldsm4(unsigned (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((unsigned)__cvta_generic_to_shared(p)));
}

// A += A' A(P, .) from the digits: a 64 x 64 tile per CTA of four warps (32 x 32
// each), every digit of the tile's rows and columns in shared memory.
constexpr int kBiGemmBytes = 2 * kBiSlices * kBiTile * kBiPitch * 2;
__global__ void __launch_bounds__(128) k_bi_gemm(double* __restrict__ A, int n, BiWork w, const int* __restrict__ info) {
  if (info[0] != 0) return;
  extern __shared__ __align__(16) uint16_t gsm[];
  uint16_t* SA = gsm;
  uint16_t* SB = SA + kBiSlices * kBiTile * kBiPitch;
  const int row0 = blockIdx.x * kBiTile, col0 = blockIdx.y * kBiTile;
  const int tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  // 7 slices x 64 rows x 4 chunks of 16 bytes each
  for (int e = tid; e < kBiSlices * kBiTile * 4; e += 128) {
    const int c = e & 3, r = (e >> 2) & (kBiTile - 1), s = e >> 8;
    const unsigned da = (unsigned)__cvta_generic_to_shared(SA + (s * kBiTile + r) * kBiPitch + c * 8);
    const unsigned db = (unsigned)__cvta_generic_to_shared(SB + (s * kBiTile + r) * kBiPitch + c * 8);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(da),
                 "l"(w.da + ((size_t)s * w.np + row0 + r) * kBiNb + c * 8));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(db),
                 "l"(w.db + ((size_t)s * w.np + col0 + r) * kBiNb + c * 8));
  }
  asm volatile("cp.async.commit_group;\n" ::);
  asm volatile("cp.async.wait_group 0;\n" ::);
  __syncthreads();
  const int wm = (wp & 1) * 32, wn = (wp >> 1) * 32;
  long long T[2][4][4];  // sums in units of 2^-54
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) T[i][j][c] = 0;
  // ldmatrix rows: A 16 x 16 blocks (lane & 15, half lane >> 4); B two 8-column blocks by two halves
  const uint16_t* pa = SA + (wm + (lane & 15)) * kBiPitch + (lane >> 4) * 8;
  const uint16_t* pb = SB + (wn + (lane & 7) + ((lane >> 4) << 3)) * kBiPitch + ((lane >> 3) & 1) * 8;
#pragma unroll 1
  for (int d = 0; d < 8; ++d) {
    float acc[2][4][4] = {};
#pragma unroll 1
    for (int i = max(0, d - (kBiSlices - 1)); i <= min(d, kBiSlices - 1); ++i) {
      const uint16_t* qa = pa + i * kBiTile * kBiPitch;
      const uint16_t* qb = pb + (d - i) * kBiTile * kBiPitch;
#pragma unroll
      for (int k = 0; k < kBiNb; k += 16) {
        unsigned a[2][4], bb[2][4];
        ldsm4(a[0], qa + k);
        ldsm4(a[1], qa + 16 * kBiPitch + k);
        ldsm4(bb[0], qb + k);
        ldsm4(bb[1], qb + 16 * kBiPitch + k);
#pragma unroll
        for (int x = 0; x < 2; ++x)
#pragma unroll
          for (int y = 0; y < 4; ++y) {
            float(&c)[4] = acc[x][y];
            asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
                         "{%0,%1,%2,%3};\n"
                         : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                         : "r"(a[x][0]), "r"(a[x][1]), "r"(a[x][2]), "r"(a[x][3]), "r"(bb[y >> 1][(y & 1) * 2]),
                           "r"(bb[y >> 1][(y & 1) * 2 + 1]));
          }
      }
    }
    // weight 2^(-14 - 8 d), in units of 2^-54: 2^(40 - 8 d)
    const int up = 40 - 8 * d;
#pragma unroll
    for (int x = 0; x < 2; ++x)
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const int q = __float_as_int(acc[x][y][c] + 12582912.f) - 0x4B400000;  // exact: |acc| < 2^22
          T[x][y][c] += up >= 0 ? (long long)q << up : (long long)((q + (1 << (-up - 1))) >> -up);
        }
  }
  const int g = lane >> 2, t2 = (lane & 3) * 2;
#pragma unroll
  for (int x = 0; x < 2; ++x)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int r = row0 + wm + x * 16 + g + 8 * h;
      if (r >= n) continue;
      const int ea = w.ea[r];
#pragma unroll
      for (int y = 0; y < 4; ++y)
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          const int col = col0 + wn + y * 8 + t2 + c;
          if (col >= n) continue;
          const long long q = T[x][y][2 * h + c];
          const int es = ea + w.eb[col] - 54;
          double* o = A + r + (long)col * n;
          if (es > kBiBad / 2)
            *o = __longlong_as_double(0x7ff8000000000000ll);  // an operand was not finite
          else if (q)
            *o += scale_pow2((double)q, es);
        }
    }
}

// out(k, piv[k']) = M(piv[k], k')
__global__ void __launch_bounds__(256) k_bi_out(const double* __restrict__ M, int n, const int* __restrict__ piv,
                                                double* __restrict__ out, int ldo, const int* __restrict__ info) {
  if (info[0] != 0) return;
  for (int c = blockIdx.y; c < n; c += gridDim.y) {
    const int k = blockIdx.x * 256 + threadIdx.x;
    if (k < n) out[k + (long)piv[c] * ldo] = M[piv[k] + (long)c * n];
  }
}

}  // namespace ifmm
