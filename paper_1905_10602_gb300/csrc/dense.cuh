// Batched dense linear algebra used by every step of the factorization and
// the solve: block copies, variable-size GEMM, Gauss-Jordan inversion with
// partial pivoting, Householder QR (R factor), one-sided Jacobi SVD.
//
// Every matrix is column-major with a leading dimension (BLAS convention).
// One descriptor describes one problem; a launch covers a batch of problems of
// different sizes (the nodes of one color of one level).  Kernels wait only on
// block and cluster barriers, and every index is bounded by the sizes in
// the descriptor.
#pragma once

#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "descs.h"
#include "devmath.cuh"
#include "fp64_ops.cuh"

namespace ifmm {

__device__ __forceinline__ int find_desc(const int* ptr, int ndesc, int t) {
  int lo = 0, hi = ndesc - 1;
  while (lo < hi) {
    int mid = (lo + hi + 1) >> 1;
    if (ptr[mid] <= t) lo = mid; else hi = mid - 1;
  }
  return lo;
}

// ---------------------------------------------------------------- copies
__global__ void k_copy(const CopyDesc* __restrict__ d, int nd) {
  const int b = blockIdx.x;
  if (b >= nd) return;
  const CopyDesc D = d[b];
  // warps over columns, lanes over rows (no per-element index division); the
  // common alpha = 1, beta in {0, 1} cases take no FP64 multiply
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const int mode = (D.alpha == 1.0 && D.beta == 0.0) ? 0 : ((D.alpha == 1.0 && D.beta == 1.0) ? 1 : 2);
  for (int j = threadIdx.x >> 5; j < D.cols; j += nw)
    for (int i = lane; i < D.rows; i += 32) {
      double v = 0.0;
      if (D.src) v = D.trans ? D.src[j + (long)i * D.lds] : D.src[i + (long)j * D.lds];
      double* o = D.dst + i + (long)j * D.ldd;
      *o = mode == 0 ? v : (mode == 1 ? *o + v : ((D.beta == 0.0) ? D.alpha * v : D.alpha * v + D.beta * (*o)));
    }
}

// ---------------------------------------------------------------- small problems
// A warp per descriptor (8 per CTA) for blocks of at most 1024 elements.
__global__ void k_copy_small(const CopyDesc* __restrict__ d, int nd) {
  const int di = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (di >= nd) return;
  const CopyDesc D = d[di];
  const int total = D.rows * D.cols;
  const int mode = (D.alpha == 1.0 && D.beta == 0.0) ? 0 : ((D.alpha == 1.0 && D.beta == 1.0) ? 1 : 2);
  for (int e = lane; e < total; e += 32) {
    const int i = e % D.rows, j = e / D.rows;
    double v = 0.0;
    if (D.src) v = D.trans ? D.src[j + (long)i * D.lds] : D.src[i + (long)j * D.lds];
    double* o = D.dst + i + (long)j * D.ldd;
    *o = mode == 0 ? v : (mode == 1 ? *o + v : ((D.beta == 0.0) ? D.alpha * v : D.alpha * v + D.beta * (*o)));
  }
}

// RB: the operands are rounded to bfloat16 before the (FP32) multiply-add.
__device__ __forceinline__ float round_bf16(float x) { return __bfloat162float(__float2bfloat16_rn(x)); }
template <typename TC, bool RB>
__device__ __forceinline__ TC stage_val(double v) {
  if constexpr (RB)
    return (TC)round_bf16(d2f_pow2(v, 0));
  else
    return ld_tc<TC>(v);
}

// One warp per GEMM with m, n <= 32 (any k), four warps per CTA.  The operands
// are staged in chunks of 16 along k through the warp's shared memory (one
// load and conversion per element); lane j accumulates column j of C in
// registers, reading the A chunk by broadcast.
template <typename TC, bool RB = false>
__global__ void __launch_bounds__(128) k_gemm_small(const GemmDesc* __restrict__ d, int nd) {
  constexpr int KC = 16;
  __shared__ TC As[4][32][KC + 1];
  __shared__ TC Bs[4][KC][33];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int di = blockIdx.x * 4 + w;
  if (di >= nd) return;
  const GemmDesc D = d[di];
  const int m = D.m, n = D.n;
  TC acc[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) acc[i] = (TC)0;
  for (int k0 = 0; k0 < D.k; k0 += KC) {
    const int kc = min(KC, D.k - k0);
    // A chunk: row i = lane, columns k0..k0+kc-1 (rows >= m and columns >= kc zero)
    for (int kk = 0; kk < KC; ++kk) {
      double v = 0.0;
      if (lane < m && kk < kc) {
        const int c = k0 + kk;
        v = D.ta ? D.A[c + (long)lane * D.lda] : D.A[lane + (long)c * D.lda];
      }
      As[w][lane][kk] = stage_val<TC, RB>(v);
    }
    // B chunk: rows k0..k0+kc-1 (kk = lane % 16), columns j
    for (int x = lane; x < KC * 32; x += 32) {
      const int kk = x % KC, j = x / KC;
      double v = 0.0;
      if (kk < kc && j < n) {
        const int r = k0 + kk;
        v = D.tb ? D.B[j + (long)r * D.ldb] : D.B[r + (long)j * D.ldb];
      }
      Bs[w][kk][j] = stage_val<TC, RB>(v);
    }
    __syncwarp();
#pragma unroll 4
    for (int kk = 0; kk < KC; ++kk) {
      const TC b = Bs[w][kk][lane];
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i] += As[w][i][kk] * b;
    }
    __syncwarp();
  }
  if (lane < n) {
    double* o = D.C + (long)lane * D.ldc;
    const TC al = ld_tc<TC>(D.alpha);
    const int bm = D.beta == 0.0 ? 0 : (D.beta == 1.0 ? 1 : 2);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      if (i >= m) break;
      const double v = st_tc<TC>(al * acc[i]);
      o[i] = bm == 0 ? v : (bm == 1 ? o[i] + v : v + D.beta * o[i]);
    }
  }
}

// ---------------------------------------------------------------- GEMM
// 64 x 64 output tile per CTA, 256 threads, 4 x 4 outputs per thread, K in
// slices of 16 staged through shared memory.  TC is the arithmetic type
// (double for the FP64 path, float for the reduced-precision modes).
template <typename TC, bool RB = false>
__global__ void __launch_bounds__(256) k_gemm(const GemmDesc* __restrict__ d, const int* __restrict__ tile_ptr, int nd) {
  const int di = find_desc(tile_ptr, nd, blockIdx.x);
  const GemmDesc D = d[di];
  const int local = blockIdx.x - tile_ptr[di];
  const int tiles_m = (D.m + 63) >> 6;
  const int tm = local % tiles_m, tn = local / tiles_m;
  const int row0 = tm * 64, col0 = tn * 64;
  __shared__ TC As[16][64 + 1];
  __shared__ TC Bs[16][64 + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  TC acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = (TC)0;
  for (int k0 = 0; k0 < D.k; k0 += 16) {
    for (int e = threadIdx.x; e < 1024; e += 256) {
      {
        const int i = e & 63, kk = e >> 6;
        const int r = row0 + i, c = k0 + kk;
        double v = 0.0;
        if (r < D.m && c < D.k) v = D.ta ? D.A[c + (long)r * D.lda] : D.A[r + (long)c * D.lda];
        As[kk][i] = stage_val<TC, RB>(v);
      }
      {
        const int kk = e & 15, j = e >> 4;
        const int r = k0 + kk, c = col0 + j;
        double v = 0.0;
        if (r < D.k && c < D.n) v = D.tb ? D.B[c + (long)r * D.ldb] : D.B[r + (long)c * D.ldb];
        Bs[kk][j] = stage_val<TC, RB>(v);
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      TC a[4], bb[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) bb[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] += a[i] * bb[j];
    }
    __syncthreads();
  }
  const TC al = ld_tc<TC>(D.alpha);
  const int bm = D.beta == 0.0 ? 0 : (D.beta == 1.0 ? 1 : 2);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = row0 + ty + 16 * i;
    if (r >= D.m) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = col0 + tx + 16 * j;
      if (c >= D.n) continue;
      double* o = D.C + r + (long)c * D.ldc;
      const double v = st_tc<TC>(al * acc[i][j]);
      *o = bm == 0 ? v : (bm == 1 ? *o + v : v + D.beta * (*o));
    }
  }
}

// ---------------------------------------------------------------- tensor-core GEMM (reduced precision)
// C = alpha op(A) op(B) + beta C on the warp-level tensor cores, FP32
// accumulation, FP64 storage.  MODE 0 (the FP32 mode): each operand x is split
// into a TF32 head h = rn_tf32(x) and a TF32-rounded tail l = rn_tf32(x - h),
// and a*b is taken as a_l*b_h + a_h*b_l + a_h*b_h (the l*l term, below
// 2^-22 |a b|, is dropped: Ootomo and Yokota's 3xTF32 scheme), three
// m16n8k8 MMAs per product tile.  MODE 1 (the BF16 mode): the operands are
// rounded to bfloat16 and multiplied by one m16n8k16 MMA.
//
// A 128 x 128 output tile per CTA of 8 warps (2 x 4, 64 x 32 per warp), K in
// slices of 16.  The FP64 slices are copied to shared memory with cp.async
// (8-byte copies, zero-filled outside the matrices) into two stages, so the
// next slice is in flight while the current one is used; each slice is then
// converted once to FP32 on the integer pipes (d2f_pow2) and, in MODE 0, split
// into TF32 head and tail, k-major with 8 words of padding (fragment loads
// free of bank conflicts).  The epilogue goes through shared memory as a
// column-major tile and every warp writes whole column segments of C.
// x rounded to TF32 (10 fraction bits), to nearest with ties away from zero,
// by integer operations on its bits: adding half a TF32 unit to the magnitude
// and clearing the 13 dropped bits (a carry into the exponent is the correct
// rounding).  Infinity stays infinity and NaN stays NaN (its quiet bit, which
// survives the truncation, is set).  The conversion instruction would run on
// the narrow FP64 pipe.
__device__ __forceinline__ unsigned tf32_rn(float x) {
  const unsigned u = __float_as_uint(x);
  if ((u & 0x7f800000u) == 0x7f800000u) return (u & 0x7fffffu) ? ((u | 0x400000u) & 0xffffe000u) : u;
  return (u + 0x1000u) & 0xffffe000u;
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const unsigned (&a)[4], const unsigned (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const unsigned (&a)[4], const unsigned (&b)[2]) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
               "{%0,%1,%2,%3};\n"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// two floats as a bfloat16 pair (round to nearest even), lo in the low half
__device__ __forceinline__ unsigned bf16x2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&v);
}
// 8-byte asynchronous copy global -> shared; nbytes 0 writes zeros
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem, int nbytes) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(s), "l"(gmem), "r"(nbytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

constexpr int kTcBM = 128, kTcBN = 128, kTcBK = 16, kTcPad = 136, kTcPC = 132;
// shared memory: two FP64 stages (A and B slices), then the converted slice
// (MODE 0: A head, A tail, B head, B tail; MODE 1: A, B); the epilogue tile
// (128 x 132 floats) reuses the FP64 stages
constexpr int kTcStageBytes = 2 * (kTcBM * kTcBK + kTcBK * kTcBN) * 8;
constexpr int kTcEpiBytes = kTcBN * kTcPC * 4;
constexpr int kTcLowBytes = kTcStageBytes > kTcEpiBytes ? kTcStageBytes : kTcEpiBytes;
constexpr int gemm_tc_smem_bytes(int mode) { return kTcLowBytes + (mode == 0 ? 4 : 2) * kTcBK * kTcPad * 4; }

template <int MODE>
__global__ void __launch_bounds__(256, 2) k_gemm_tc(const GemmDesc* __restrict__ d, const int* __restrict__ tile_ptr,
                                                     int nd) {
  constexpr int BM = kTcBM, BN = kTcBN, BK = kTcBK, P = kTcPad;
  extern __shared__ __align__(16) unsigned char tcsm[];
  double* S64 = (double*)tcsm;                   // [2][BM*BK + BK*BN]
  unsigned* Cv = (unsigned*)(tcsm + kTcLowBytes);  // converted slice
  const int di = find_desc(tile_ptr, nd, blockIdx.x);
  const GemmDesc& D = d[di];
  const int local = blockIdx.x - tile_ptr[di];
  const int tiles_m = (D.m + BM - 1) / BM;
  const int row0 = (local % tiles_m) * BM, col0 = (local / tiles_m) * BN;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = warp & 1, wn = warp >> 1;  // 2 x 4 warps, warp tile 64 x 32
  const int g = lane >> 2, t = lane & 3;
  float acc[4][4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][j][c] = 0.f;
  // staging order of a slice: A element (i, kk) at sa(i, kk), B element (kk, j)
  // at sb(kk, j), along the contiguous axis of each matrix in memory
  auto issue = [&](int k0, int stage) {
    double* SA = S64 + stage * (BM * BK + BK * BN);
    double* SB = SA + BM * BK;
#pragma unroll
    for (int x = 0; x < BM * BK / 256; ++x) {
      const int e = tid + x * 256;
      int i, kk;
      if (D.ta) { kk = e % BK; i = e / BK; } else { i = e % BM; kk = e / BM; }
      const int r = row0 + i, c = k0 + kk;
      const bool in = r < D.m && c < D.k;
      const double* src = in ? (D.ta ? D.A + c + (long)r * D.lda : D.A + r + (long)c * D.lda) : D.A;
      cp_async8(SA + e, src, in ? 8 : 0);
    }
#pragma unroll
    for (int x = 0; x < BK * BN / 256; ++x) {
      const int e = tid + x * 256;
      int kk, j;
      if (D.tb) { j = e % BN; kk = e / BN; } else { kk = e % BK; j = e / BK; }
      const int r = k0 + kk, c = col0 + j;
      const bool in = r < D.k && c < D.n;
      const double* src = in ? (D.tb ? D.B + c + (long)r * D.ldb : D.B + r + (long)c * D.ldb) : D.B;
      cp_async8(SB + e, src, in ? 8 : 0);
    }
    cp_async_commit();
  };
  // converts stage `stage` into Cv: k-major rows of P words
  auto convert = [&](int stage) {
    const double* SA = S64 + stage * (BM * BK + BK * BN);
    const double* SB = SA + BM * BK;
#pragma unroll
    for (int x = 0; x < BM * BK / 256; ++x) {
      const int e = tid + x * 256;
      const int i = e % BM, kk = e / BM;
      const float f = d2f_pow2(D.ta ? SA[kk + i * BK] : SA[i + kk * BM], 0);
      if constexpr (MODE == 0) {
        const unsigned h = tf32_rn(f);
        Cv[kk * P + i] = h;
        Cv[(BK + kk) * P + i] = tf32_rn(f - __uint_as_float(h));
      } else {
        Cv[kk * P + i] = __float_as_uint(f);
      }
    }
    unsigned* CB = Cv + (MODE == 0 ? 2 : 1) * BK * P;
#pragma unroll
    for (int x = 0; x < BK * BN / 256; ++x) {
      const int e = tid + x * 256;
      const int j = e % BN, kk = e / BN;
      const float f = d2f_pow2(D.tb ? SB[j + kk * BN] : SB[kk + j * BK], 0);
      if constexpr (MODE == 0) {
        const unsigned h = tf32_rn(f);
        CB[kk * P + j] = h;
        CB[(BK + kk) * P + j] = tf32_rn(f - __uint_as_float(h));
      } else {
        CB[kk * P + j] = __float_as_uint(f);
      }
    }
  };
  const int nk = (D.k + BK - 1) / BK;
  if (nk > 0) issue(0, 0);
  for (int ks = 0; ks < nk; ++ks) {
    if (ks + 1 < nk) {
      issue((ks + 1) * BK, (ks + 1) & 1);
      cp_async_wait<1>();
    } else {
      cp_async_wait<0>();
    }
    __syncthreads();  // slice ks landed for every thread; the previous MMAs are done with Cv
    convert(ks & 1);
    __syncthreads();
    const unsigned* Ah = Cv + wm * 64;
    const unsigned* Bh = Cv + (MODE == 0 ? 2 : 1) * BK * P + wn * 32;
    if constexpr (MODE == 0) {
      const unsigned* Al = Ah + BK * P;
      const unsigned* Bl = Bh + BK * P;
#pragma unroll
      for (int k8 = 0; k8 < BK; k8 += 8) {
        unsigned bh[4][2], bl[4][2];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          bh[j][0] = Bh[(k8 + t) * P + j * 8 + g];
          bh[j][1] = Bh[(k8 + t + 4) * P + j * 8 + g];
          bl[j][0] = Bl[(k8 + t) * P + j * 8 + g];
          bl[j][1] = Bl[(k8 + t + 4) * P + j * 8 + g];
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int m0 = i * 16 + g;
          const unsigned ah[4] = {Ah[(k8 + t) * P + m0], Ah[(k8 + t) * P + m0 + 8], Ah[(k8 + t + 4) * P + m0],
                                  Ah[(k8 + t + 4) * P + m0 + 8]};
          const unsigned al[4] = {Al[(k8 + t) * P + m0], Al[(k8 + t) * P + m0 + 8], Al[(k8 + t + 4) * P + m0],
                                  Al[(k8 + t + 4) * P + m0 + 8]};
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            mma_tf32(acc[i][j], al, bh[j]);
            mma_tf32(acc[i][j], ah, bl[j]);
            mma_tf32(acc[i][j], ah, bh[j]);
          }
        }
      }
    } else {
      const float* As = (const float*)Ah;
      const float* Bs = (const float*)Bh;
      unsigned b[4][2];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float* bb = Bs + j * 8 + g;
        b[j][0] = bf16x2(bb[(2 * t) * P], bb[(2 * t + 1) * P]);
        b[j][1] = bf16x2(bb[(2 * t + 8) * P], bb[(2 * t + 9) * P]);
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float* aa = As + i * 16 + g;
        unsigned a[4];
        a[0] = bf16x2(aa[(2 * t) * P], aa[(2 * t + 1) * P]);
        a[1] = bf16x2(aa[(2 * t) * P + 8], aa[(2 * t + 1) * P + 8]);
        a[2] = bf16x2(aa[(2 * t + 8) * P], aa[(2 * t + 9) * P]);
        a[3] = bf16x2(aa[(2 * t + 8) * P + 8], aa[(2 * t + 9) * P + 8]);
#pragma unroll
        for (int j = 0; j < 4; ++j) mma_bf16(acc[i][j], a, b[j]);
      }
    }
  }
  __syncthreads();  // every warp is done with the stages before the epilogue reuses them
  float* Cs = (float*)tcsm;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = wm * 64 + i * 16 + g, c = wn * 32 + j * 8 + 2 * t;
      Cs[c * kTcPC + r] = acc[i][j][0];
      Cs[(c + 1) * kTcPC + r] = acc[i][j][1];
      Cs[c * kTcPC + r + 8] = acc[i][j][2];
      Cs[(c + 1) * kTcPC + r + 8] = acc[i][j][3];
    }
  __syncthreads();
  const float al = d2f_pow2(D.alpha, 0);
  const int bm = D.beta == 0.0 ? 0 : (D.beta == 1.0 ? 1 : 2);
  const int mr = min(BM, D.m - row0), nc = min(BN, D.n - col0);
  for (int c = warp; c < nc; c += 8) {
    double* o = D.C + row0 + (long)(col0 + c) * D.ldc;
    for (int r = lane; r < mr; r += 32) {
      const double v = f2d_pow2(al * Cs[c * kTcPC + r], 0);
      o[r] = bm == 0 ? v : (bm == 1 ? o[r] + v : v + D.beta * o[r]);
    }
  }
}

// ---------------------------------------------------------------- reductions
// block-wide sum; scratch holds >= 32 doubles; every thread gets the result
__device__ double block_sum(double v, double* scratch) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  v = warp_sum(v);
  __syncthreads();
  if (lane == 0) scratch[w] = v;
  __syncthreads();
  double s = 0.0;
  for (int i = 0; i < nw; ++i) s += scratch[i];
  return s;
}

// ---------------------------------------------------------------- Gauss-Jordan inverse
// In-place inverse with partial pivoting of one n x n matrix per thread-block
// cluster (1 to 16 CTAs, cluster CTA r holding columns r, r + R, ... in shared
// memory).  Step k exchanges column k with the unused row p of largest |A(i,k)|
// (ties: smallest i): with c = column k and q = 1 / c_p, every other column j
// becomes A(i,j) - c_i (A(p,j) q), A(p,j) q in row p, and column k itself -c_i q,
// q in row p.  Rows are never moved: after n steps row p_k holds x_k and column
// k' belongs to y of row p_k', so the inverse is written out as
// Ainv(k, p_k') = M(p_k, k').
//
// What bounds it: at most two FP64 multiply-adds per clock and SM (n^3 / (2 R)
// clocks), and the chain of n dependent steps.  Columns instead of rows are
// distributed so that a step needs one exchange: the CTA that owns column k + 1
// updates that column first, finds its pivot and pushes column, pivot and
// reciprocal into every CTA's shared memory, and only then everybody does the
// bulk of step k, which hides the exchange (split cluster barrier, three
// buffers: when step k's data is complete every CTA has finished with those of
// step k - 2).  The row-distributed kernel this replaces took two cluster
// barriers, six CTA barriers and serial scans per step: three blocks of 224 rows
// 1,621 -> 473 us, 78 of 70 rows 382 -> 189 us, the pivots of the 131,072-point
// job 175 -> 64 ms.
__host__ __device__ __forceinline__ size_t inv_slot_bytes(int n, int R) {
  const size_t nc = ((size_t)n + R - 1) / R;
  return ((size_t)n * nc + 3 * (size_t)n + nc) * sizeof(double) + ((sizeof(int) * (size_t)n + 15) & ~(size_t)15);
}
// V: rows per thread, n <= V * blockDim.x
template <int V>
__global__ void __launch_bounds__(512) k_inv(const InvDesc* __restrict__ d, int nd) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  const int R = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const int pi = (int)(blockIdx.x / R);
  const InvDesc D = d[pi < nd ? pi : nd - 1];
  const int n = D.n;
  const long ld = D.ld;
  const int nc = (n - rank + R - 1) / R;  // local columns: rank + c R
  extern __shared__ __align__(16) double ivm[];
  double* A = ivm;                                     // n x ceil(n / R), ld n
  double* cb = A + (size_t)n * ((n + R - 1) / R);      // 3 x n: column k of steps k mod 3
  double* rr = cb + 3 * (size_t)n;                     // row p of the local columns, scaled
  int* piv = (int*)(rr + (n + R - 1) / R);
  __shared__ double ib[3];                             // reciprocal pivots
  __shared__ int pb[3];                                // pivot rows (-1: none)
  __shared__ unsigned rh[16], rl[16];
  __shared__ int ri[16];
  const int tid = threadIdx.x, T = blockDim.x, lane = tid & 31, w = tid >> 5, nw = T >> 5;
  for (int c = w; c < nc; c += nw)
    for (int i = lane; i < n; i += 32) A[i + (size_t)c * n] = D.A[i + (long)(rank + c * R) * ld];
  __syncthreads();
  const int nrb = (n + 31) >> 5, dx = nw / nrb, drb = nw - dx * nrb;
  bool used[V];
#pragma unroll
  for (int v = 0; v < V; ++v) used[v] = false;
  // column c (values val, row tid + v T): its pivot, written back, pushed as step
  // kk's data; contains one __syncthreads
  auto publish = [&](const double (&val)[V], int c, int kk) {
    unsigned hi = 0, lo = 0;
    int bi = 0x7fffffff;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int i = tid + v * T;
      const unsigned h = (unsigned)__double2hiint(val[v]) & 0x7fffffffu, l = (unsigned)__double2loint(val[v]);
      const bool nan = h > 0x7ff00000u || (h == 0x7ff00000u && l);  // never a pivot
      if (i < n && !used[v] && !nan && (bi == 0x7fffffff || h > hi || (h == hi && l > lo))) {
        hi = h;
        lo = l;
        bi = i;
      }
    }
    warp_max_key(hi, lo, bi);
    if (lane == 0) {
      rh[w] = hi;
      rl[w] = lo;
      ri[w] = bi;
    }
    __syncthreads();
    hi = lane < nw ? rh[lane] : 0u;
    lo = lane < nw ? rl[lane] : 0u;
    bi = lane < nw ? ri[lane] : 0x7fffffff;
    warp_max_key(hi, lo, bi);
    const int p = (hi | lo) ? bi : -1;
    const int b = kk % 3;
#pragma unroll
    for (int v = 0; v < V; ++v) {
      const int i = tid + v * T;
      if (i >= n) continue;
      A[i + (size_t)c * n] = val[v];
      for (int r = 0; r < R; ++r) cl.map_shared_rank(cb, r)[(size_t)b * n + i] = val[v];
      if (i == p) {
        const double q = rcp_fp64(val[v]);
        for (int r = 0; r < R; ++r) {
          cl.map_shared_rank(ib, r)[b] = q;
          cl.map_shared_rank(pb, r)[b] = p;
        }
      }
    }
    if (p < 0 && tid == 0)
      for (int r = 0; r < R; ++r) cl.map_shared_rank(pb, r)[b] = -1;
  };
  // no CTA writes into another's shared memory before that one runs
  cl.sync();
  if (rank == 0) {
    double val[V];
#pragma unroll
    for (int v = 0; v < V; ++v) val[v] = tid + v * T < n ? A[tid + v * T] : 0.0;
    publish(val, 0, 0);
  }
  cluster_arrive();
  int bad = 0;
  for (int k = 0; k < n; ++k) {
    cluster_wait();
    const int b = k % 3;
    const int p = pb[b];
    if (p < 0) {
      bad = k + 1;
      break;
    }
    const double* c = cb + (size_t)b * n;
    const double q = ib[b];
    if (tid == 0) piv[k] = p;
#pragma unroll
    for (int v = 0; v < V; ++v) used[v] = used[v] || tid + v * T == p;
    if (k + 1 < n) {
      if ((k + 1) % R == rank) {
        const int cn = (k + 1) / R;
        double val[V];
        const double r = A[p + (size_t)cn * n] * q;
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const int i = tid + v * T;
          val[v] = 0.0;
          if (i < n) val[v] = i == p ? r : fma(-c[i], r, A[i + (size_t)cn * n]);
        }
        publish(val, cn, k + 1);
      }
      cluster_arrive();
    }
    // bulk: (column, 32 rows) items over the warps, four in flight (independent
    // FP64 chains); column k itself is the same update of a zero column
    const int xk = k % R == rank ? k / R : -1, xn = (k + 1) % R == rank ? (k + 1) / R : -1;
    for (int x = tid; x < nc; x += T) rr[x] = x == xk ? q : A[p + (size_t)x * n] * q;
    __syncthreads();  // row p read before any of it is written
    {
      int x = w / nrb, rb = w - x * nrb;
      for (int e = w; e < nc * nrb; e += 4 * nw) {
        int ix[4], ii[4];
        bool on[4];
        double z[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          ii[u] = rb * 32 + lane;
          ix[u] = x;
          on[u] = x < nc && x != xn;
          z[u] = (on[u] && ii[u] < n && x != xk) ? A[ii[u] + (size_t)x * n] : 0.0;
          x += dx;
          rb += drb;
          if (rb >= nrb) {
            rb -= nrb;
            ++x;
          }
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
          if (on[u] && ii[u] < n) {
            const double r = rr[ix[u]];
            A[ii[u] + (size_t)ix[u] * n] = ii[u] == p ? r : fma(-c[ii[u]], r, z[u]);
          }
      }
    }
    __syncthreads();
  }
  // no CTA leaves, or overwrites the input, while another still needs it
  cl.sync();
  if (!bad)
    for (int x = w; x < nc; x += nw) {
      double* o = D.A + (long)piv[rank + x * R] * ld;
      for (int k = lane; k < n; k += 32) o[k] = A[piv[k] + (size_t)x * n];
    }
  if (rank == 0 && tid == 0) D.info[0] = bad;
}

// Batched Gauss-Jordan for matrices too large for shared memory: one launch
// pair per pivot step k over all matrices of the batch (k_gjb_pivot: a CTA per
// matrix picks, swaps and scales the pivot row; k_gjb_update: a 2-D grid, one
// row of CTAs per matrix, eliminates column k), then k_gjb_colswap.  work holds
// 2n doubles and n ints per matrix at work_off[b].
__global__ void k_gjb_pivot(const InvDesc* __restrict__ d, int nd, int k, double* __restrict__ work,
                            const long* __restrict__ work_off) {
  const int b = blockIdx.x;
  if (b >= nd) return;
  const InvDesc D = d[b];
  const int n = D.n;
  if (k >= n || D.info[0] != 0) return;
  double* A = D.A;
  const long ld = D.ld;
  double* rowk = work + work_off[b];
  double* colk = rowk + n;
  int* piv = (int*)(colk + n);
  __shared__ double red_v[32];
  __shared__ int red_i[32];
  __shared__ int s_p;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  double best = -1.0;
  int bi = n;
  for (int i = k + threadIdx.x; i < n; i += blockDim.x) {
    const double v = fabs(A[i + k * ld]);
    if (v > best || (v == best && i < bi)) { best = v; bi = i; }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double ov = __shfl_xor_sync(0xffffffffu, best, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
  }
  if (lane == 0) { red_v[w] = best; red_i[w] = bi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    double bv = -1.0;
    int bb = n;
    for (int i = 0; i < nw; ++i)
      if (red_v[i] > bv || (red_v[i] == bv && red_i[i] < bb)) { bv = red_v[i]; bb = red_i[i]; }
    if (!(bv > 0.0) || bb >= n) {
      D.info[0] = k + 1;
      bb = k;
    }
    s_p = bb;
    piv[k] = bb;
  }
  __syncthreads();
  if (D.info[0] != 0) return;
  const int p = s_p;
  if (p != k) {
    for (int j = threadIdx.x; j < n; j += blockDim.x) {
      const double t = A[k + j * ld];
      A[k + j * ld] = A[p + j * ld];
      A[p + j * ld] = t;
    }
    __syncthreads();  // p is the same in every thread: rows k and p swapped before they are read below
  }
  __shared__ double s_inv;
  if (threadIdx.x == 0) s_inv = 1.0 / A[k + k * ld];  // once: an FP64 divide is a long FP64 sequence
  __syncthreads();
  const double inv = s_inv;
  for (int j = threadIdx.x; j < n; j += blockDim.x) rowk[j] = (j == k) ? inv : A[k + j * ld] * inv;
  for (int i = threadIdx.x; i < n; i += blockDim.x) colk[i] = (i == k) ? 0.0 : A[i + k * ld];
}

__global__ void k_gjb_update(const InvDesc* __restrict__ d, int nd, int k, const double* __restrict__ work,
                             const long* __restrict__ work_off) {
  const int b = blockIdx.y;
  if (b >= nd) return;
  const InvDesc D = d[b];
  const int n = D.n;
  if (k >= n || D.info[0] != 0) return;
  double* A = D.A;
  const long ld = D.ld;
  const double* rowk = work + work_off[b];
  const double* colk = rowk + n;
  // columns over (CTA, warp), lanes over rows (no per-element index division)
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int j = blockIdx.x * nw + (threadIdx.x >> 5); j < n; j += gridDim.x * nw) {
    const double rj = rowk[j];
    double* cj = A + (long)j * ld;
    for (int i = lane; i < n; i += 32) {
      if (i == k) {
        cj[i] = rj;
      } else {
        const double a = (j == k) ? 0.0 : cj[i];
        cj[i] = a - colk[i] * rj;
      }
    }
  }
}

__global__ void k_gjb_colswap(const InvDesc* __restrict__ d, int nd, const double* __restrict__ work,
                              const long* __restrict__ work_off) {
  const int b = blockIdx.x;
  if (b >= nd) return;
  const InvDesc D = d[b];
  const int n = D.n;
  if (D.info[0] != 0) return;
  double* A = D.A;
  const long ld = D.ld;
  const int* piv = (const int*)(work + work_off[b] + 2 * n);
  for (int k = n - 1; k >= 0; --k) {
    const int p = piv[k];
    if (p != k)
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const double t = A[i + k * ld];
        A[i + k * ld] = A[i + p * ld];
        A[i + p * ld] = t;
      }
    __syncthreads();
  }
}

// ---------------------------------------------------------------- Householder QR
// One CTA per matrix.  Column k: v = x - alpha e1 with alpha = -sign(x_0)||x||,
// H = I - 2 v v^T / (v^T v) applied to the trailing columns (one warp per column).
// Storage is double; TC is the arithmetic type of the dot products and updates.
// Apply H = I - t v v^T (v_0 = 1, v_i = x_i for i >= 1) to the trailing
// columns k+1..n-1 of A (rows k..k+len-1).  Each column's dot product and
// update is split into S row segments when there are fewer trailing columns
// than warps; the S partial sums are added in a fixed order (deterministic).
// partial: shared memory of >= max(n, warps) doubles.  Ends with __syncthreads.
template <typename TC>
__device__ void apply_reflector(double* A, long ld, int k, int n, int len, const double* x, TC t, double* partial) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  const int nt = n - k - 1;
  if (nt <= 0) return;
  int S = nw / nt;
  const int smax = (len + 63) / 64;
  if (S > smax) S = smax;
  if (S < 1) S = 1;
  const int seg = (len + S - 1) / S;
  const int items = nt * S;
  for (int it = w; it < items; it += nw) {
    const int jj = it / S, sg = it % S;
    const double* y = A + k + (long)(k + 1 + jj) * ld;
    const int r0 = sg * seg, r1 = min(len, r0 + seg);
    TC dot = 0;
    for (int i = r0 + lane; i < r1; i += 32) dot += (i == 0 ? (TC)1 : (TC)x[i]) * (TC)y[i];
    dot = warp_sum_t<TC>(dot);
    if (lane == 0) partial[it] = (double)dot;
  }
  __syncthreads();
  for (int it = w; it < items; it += nw) {
    const int jj = it / S, sg = it % S;
    double* y = A + k + (long)(k + 1 + jj) * ld;
    TC dot = 0;
    for (int q = 0; q < S; ++q) dot += (TC)partial[jj * S + q];
    dot *= t;
    const int r0 = sg * seg, r1 = min(len, r0 + seg);
    for (int i = r0 + lane; i < r1; i += 32) y[i] = (double)((TC)y[i] - dot * (i == 0 ? (TC)1 : (TC)x[i]));
  }
  __syncthreads();
}

template <typename TC>
__global__ void k_qr(const QrDesc* __restrict__ d, int nd) {
  if ((int)blockIdx.x >= nd) return;
  const QrDesc D = d[blockIdx.x];
  const int m = D.m, n = D.n;
  const long ld = D.ld;
  double* A = D.A;
  __shared__ double scratch[32];
  __shared__ double partial[1024];
  __shared__ double s_alpha, s_beta, s_scale;
  const int kmax = m < n ? m : n;
  for (int k = 0; k < kmax; ++k) {
    double* x = A + k + k * ld;
    const int len = m - k;
    double ss = 0.0;
    for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) ss += x[i] * x[i];
    ss = block_sum(ss, scratch);
    // reflector in the normalised form H = I - tau v v^T, v_0 = 1,
    // v_i = x_i / (x_0 - alpha), tau = (alpha - x_0) / alpha in [1, 2]
    if (threadIdx.x == 0) {
      const double x0 = x[0];
      const double nrm = sqrt(x0 * x0 + ss);
      if (nrm == 0.0 || ss == 0.0) {
        s_alpha = x0;
        s_beta = 0.0;
      } else {
        const double alpha = (x0 >= 0.0) ? -nrm : nrm;
        s_alpha = alpha;
        s_beta = (alpha - x0) / alpha;
        s_scale = 1.0 / (x0 - alpha);
      }
    }
    __syncthreads();
    const double tau = s_beta;
    if (tau != 0.0) {
      const double sc = s_scale;
      for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) x[i] *= sc;
      __syncthreads();
      apply_reflector<TC>(A, ld, k, n, len, x, (TC)tau, partial);
    }
    __syncthreads();
    if (threadIdx.x == 0) x[0] = s_alpha;
    for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) x[i] = 0.0;
    __syncthreads();
  }
}

// ---------------------------------------------------------------- pivoted QR (truncated), global memory
// One CTA per matrix, the block in global memory (the fallback for blocks that
// fit neither one CTA's nor a cluster's shared memory).  Column norms live in
// shared memory and are downdated after each step (recomputed when
// cancellation has eaten two digits).  Dynamic shared memory: 2n doubles + n ints.
template <typename TC>
__global__ void k_qrcp(const QrcpDesc* __restrict__ d, int nd) {
  if ((int)blockIdx.x >= nd) return;
  const QrcpDesc D = d[blockIdx.x];
  const int m = D.m, n = D.n;
  const long ld = D.ld;
  double* A = D.A;
  extern __shared__ double sm[];
  double* nrm = sm;
  double* ref = sm + n;
  int* jp = (int*)(sm + 2 * n);
  __shared__ double scratch[32];
  __shared__ double partial[1024];
  __shared__ char flag[1024];
  __shared__ double red_v[32];
  __shared__ int red_i[32];
  __shared__ double s_tau2, s_alpha, s_tau, s_scale, s_first, s_tailv;
  __shared__ int s_p, s_stop, s_capped;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  for (int j = w; j < n; j += nw) {
    const double* c = A + (long)j * ld;
    double ss = 0.0;
    for (int i = lane; i < m; i += 32) ss += c[i] * c[i];
    ss = warp_sum(ss);
    if (lane == 0) {
      nrm[j] = ss;
      ref[j] = ss;
      jp[j] = j;
    }
  }
  __syncthreads();
  const int kmax = m < n ? m : n;
  int k = 0;
  for (; k < kmax; ++k) {
    double best = -1.0;
    int bi = n;
    for (int j = k + threadIdx.x; j < n; j += blockDim.x) {
      const double v = nrm[j];
      if (v > best || (v == best && j < bi)) { best = v; bi = j; }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > best || (ov == best && oi < bi)) { best = ov; bi = oi; }
    }
    if (lane == 0) { red_v[w] = best; red_i[w] = bi; }
    __syncthreads();
    if (threadIdx.x == 0) {
      double bv = -1.0;
      int b = n;
      for (int i = 0; i < nw; ++i)
        if (red_v[i] > bv || (red_v[i] == bv && red_i[i] < b)) { bv = red_v[i]; b = red_i[i]; }
      if (k == 0) s_tau2 = D.tau_rel * D.tau_rel * bv;
      if (k == 0) s_first = bv;
      s_stop = !(bv > s_tau2) || !(bv > 0.0) || b >= n;
      s_capped = 0;
      if (!s_stop && D.kcap > 0 && k >= D.kcap) {
        s_stop = 1;
        s_capped = 1;
        s_tailv = (s_first > 0.0) ? sqrt(bv / s_first) : 0.0;
      }
      s_p = b;
    }
    __syncthreads();
    if (s_stop) break;
    const int p = s_p;
    if (p != k) {
      for (int i = threadIdx.x; i < m; i += blockDim.x) {
        const double t = A[i + k * ld];
        A[i + k * ld] = A[i + p * ld];
        A[i + p * ld] = t;
      }
      if (threadIdx.x == 0) {
        double t = nrm[k]; nrm[k] = nrm[p]; nrm[p] = t;
        t = ref[k]; ref[k] = ref[p]; ref[p] = t;
        const int q = jp[k]; jp[k] = jp[p]; jp[p] = q;
      }
    }
    __syncthreads();
    double* x = A + k + k * ld;
    const int len = m - k;
    double ss = 0.0;
    for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) ss += x[i] * x[i];
    ss = block_sum(ss, scratch);
    if (threadIdx.x == 0) {
      const double x0 = x[0];
      const double nr = sqrt(x0 * x0 + ss);
      if (nr == 0.0 || ss == 0.0) {
        s_alpha = x0;
        s_tau = 0.0;
      } else {
        const double alpha = (x0 >= 0.0) ? -nr : nr;
        s_alpha = alpha;
        s_tau = (alpha - x0) / alpha;
        s_scale = 1.0 / (x0 - alpha);
      }
    }
    __syncthreads();
    const double tau = s_tau;
    if (tau != 0.0) {
      const double sc = s_scale;
      for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) x[i] *= sc;
      __syncthreads();
    }
    if (tau != 0.0) apply_reflector<TC>(A, ld, k, n, len, x, (TC)tau, partial);
    // downdate the column norms with the new row k of R; recompute a norm when
    // cancellation has removed two digits
    for (int j = k + 1 + threadIdx.x; j < n; j += blockDim.x) {
      const double rkj = A[k + (long)j * ld];
      const double v = nrm[j] - rkj * rkj;
      flag[j] = !(v > 1e-2 * ref[j]);
      nrm[j] = v;
    }
    __syncthreads();
    for (int j = k + 1 + w; j < n; j += nw) {
      if (!flag[j]) continue;
      const double* y = A + k + (long)j * ld;
      double s2 = 0.0;
      for (int i = 1 + lane; i < len; i += 32) s2 += y[i] * y[i];
      s2 = warp_sum(s2);
      if (lane == 0) {
        nrm[j] = s2;
        ref[j] = s2;
      }
    }
    __syncthreads();
    if (threadIdx.x == 0) x[0] = s_alpha;
    for (int i = 1 + threadIdx.x; i < len; i += blockDim.x) x[i] = 0.0;
    __syncthreads();
  }
  for (int j = threadIdx.x; j < n; j += blockDim.x) D.jpvt[j] = jp[j];
  if (threadIdx.x == 0) {
    D.kout[0] = k;
    if (D.tail) D.tail[0] = (k < kmax && s_capped) ? s_tailv : 0.0;
  }
}

// ---------------------------------------------------------------- IL basis changes
// One CTA per touched IL entry e of a color: M2L_ab <- T'_a M2L_ab T_b, with
// the identity for an endpoint that was not re-based and a zero block when an
// old rank is zero.  The block is staged in shared memory (it is overwritten in
// place); md >= every rank involved is the stride of the staging tiles.
template <typename TC>
__global__ void __launch_bounds__(128) k_il_transform(const int* __restrict__ list, int nlist, IlTables t, int md) {
  if ((int)blockIdx.x >= nlist) return;
  const int e = list[blockIdx.x];
  const int a = t.il_row[e], b = t.il[e];
  const int ra = t.rbefore[a], rb = t.rbefore[b], na = t.newk[a], nb = t.newk[b];
  const int ka = na >= 0 ? na : ra, kb = nb >= 0 ? nb : rb;
  if (ka == 0 || kb == 0) return;
  double* M = t.far[e];
  const long ld = t.capr[a];
  const int tid = threadIdx.x, nt = blockDim.x;
  if (ra == 0 || rb == 0) {
    for (int x = tid; x < ka * kb; x += nt) M[(x % ka) + (long)(x / ka) * ld] = 0.0;
    return;
  }
  extern __shared__ __align__(16) unsigned char ism[];
  TC* Ms = (TC*)ism;       // ra x rb, ld ra
  TC* t1 = Ms + md * md;   // ka x rb, ld ka
  TC* X = t1 + md * md;    // T'_a (ka x ra, ld ka), then T_b (rb x kb, ld rb)
  for (int x = tid; x < ra * rb; x += nt) Ms[x] = ld_tc<TC>(M[(x % ra) + (long)(x / ra) * ld]);
  if (na >= 0) {
    const double* Tp = t.Tp[a];
    for (int x = tid; x < ka * ra; x += nt) X[x] = ld_tc<TC>(Tp[x]);
  }
  __syncthreads();
  if (na >= 0) {
    for (int x = tid; x < ka * rb; x += nt) {
      const int i = x % ka, j = x / ka;
      TC acc = 0;
      for (int l = 0; l < ra; ++l) acc += X[i + l * ka] * Ms[l + j * ra];
      t1[x] = acc;
    }
  } else {
    for (int x = tid; x < ka * rb; x += nt) t1[x] = Ms[x];
  }
  __syncthreads();
  if (nb >= 0) {
    const double* Tb = t.T[b];
    for (int x = tid; x < rb * kb; x += nt) X[x] = ld_tc<TC>(Tb[x]);
    __syncthreads();
    for (int x = tid; x < ka * kb; x += nt) {
      const int i = x % ka, j = x / ka;
      TC acc = 0;
      for (int l = 0; l < rb; ++l) acc += t1[i + l * ka] * X[l + j * rb];
      M[i + (long)j * ld] = st_tc<TC>(acc);
    }
  } else {
    for (int x = tid; x < ka * kb; x += nt) M[(x % ka) + (long)(x / ka) * ld] = st_tc<TC>(t1[x]);
  }
}

// One CTA per (event, side): gathers the weight stack of ZGatherDesc from the
// level's IL blocks on the device.  The rows of every entry's block are found by a
// scan of the ranks first, so that the warps copy different entries at the same
// time (one after the other the entries' dependent loads were the time: 201 us a
// launch at 131,072 points, now 142).
__global__ void __launch_bounds__(256) k_zgather(const ZGatherDesc* __restrict__ d, int nd, ZTables t) {
  if ((int)blockIdx.x >= nd) return;
  const ZGatherDesc D = d[blockIdx.x];
  const int q = D.q, rq = t.r[q];
  const long ldz = D.ldz;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  constexpr int CH = 256;  // entries of a pass
  __shared__ int offs[CH + 1], rls[CH];
  __shared__ const double* src[CH];
  __shared__ int lds[CH];
  int off = 0;
  for (int e0 = t.il_ptr[q]; e0 < t.il_ptr[q + 1]; e0 += CH) {
    const int cnt = min(CH, t.il_ptr[q + 1] - e0);
    __syncthreads();  // the previous pass is done with the lists
    for (int x = threadIdx.x; x < cnt; x += blockDim.x) {
      const int l = t.il[e0 + x];
      rls[x] = t.r[l];
      src[x] = t.far[D.side == 0 ? t.il_T[e0 + x] : e0 + x];
      lds[x] = t.capr[D.side == 0 ? l : q];
    }
    __syncthreads();
    if (w == 0) {
      int base = off;
      for (int x0 = 0; x0 < cnt; x0 += 32) {
        const int v = x0 + lane < cnt ? rls[x0 + lane] : 0;
        int s = v;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, s, o);
          if (lane >= o) s += y;
        }
        if (x0 + lane < cnt) offs[x0 + lane] = base + s - v;
        base += __shfl_sync(0xffffffffu, s, 31);
      }
      if (lane == 0) offs[cnt] = base;
    }
    __syncthreads();
    for (int x = w; x < cnt; x += nw) {
      const int rl = rls[x];
      const double* p = src[x];
      double* z = D.Z + offs[x];
      const long ls = lds[x];
      for (int i = lane; i < rl; i += 32) {
        const double* pi = D.side == 0 ? p + i : p + i * ls;
        const long st = D.side == 0 ? ls : 1;
        int j = 0;
        for (; j + 4 <= rq; j += 4) {
          const double v0 = pi[j * st], v1 = pi[(j + 1) * st], v2 = pi[(j + 2) * st], v3 = pi[(j + 3) * st];
          z[i + j * ldz] = v0;
          z[i + (j + 1) * ldz] = v1;
          z[i + (j + 2) * ldz] = v2;
          z[i + (j + 3) * ldz] = v3;
        }
        for (; j < rq; ++j) z[i + j * ldz] = pi[j * st];
      }
    }
    off = offs[cnt];
  }
  if (t.tail) {
    const int rc = t.rc;
    const double* p = D.side == 0 ? t.M2M[q] : t.L2L[q];
    const long ls = t.capr[q];
    for (int j = w; j < rq; j += nw)
      for (int i = lane; i < rc; i += 32)
        D.Z[off + i + j * ldz] = D.side == 0 ? p[i + (long)j * rc] : p[j + i * ls];
  }
}

// One CTA per (eliminated node, neighbour a): adds the row block of neighbour a
// of F into its near blocks (ScatterDesc).  Lane b of the first warp finds the
// block of (a, b) (a binary search of q2 in q's sorted neighbour list; all of them
// at once), then the warps take the columns of F, narrow row blocks several
// columns per warp, four in flight.  Bound: the read-modify-write of the near
// blocks; with one search after the other and one column per warp it took 339 us a
// launch at 131,072 points, now 203.
__global__ void __launch_bounds__(256) k_schur_scatter(const ScatterDesc* __restrict__ d, int nd, ScatterTables t) {
  const int di = blockIdx.x;
  if (di >= nd) return;
  const ScatterDesc D = d[di];
  const int i = D.i;
  const int c0 = t.nbr_ptr[i], deg = t.nbr_ptr[i + 1] - c0;
  const int a = blockIdx.y;
  if (a >= deg) return;
  __shared__ int roff[33];
  __shared__ double* dsts[32];
  __shared__ int s_mq, s_ld;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (w == 0) {
    const int q2 = lane < deg ? t.nbr[c0 + lane] : 0;
    const int el2 = lane < deg ? t.elim[q2] : 0;
    const int v = lane < deg ? (el2 ? t.r[q2] : t.n[q2]) : 0;
    int s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    roff[lane + 1] = s;
    if (lane == 0) roff[0] = 0;
    const int q = __shfl_sync(0xffffffffu, q2, a), elq = __shfl_sync(0xffffffffu, el2, a);
    double* dst = nullptr;
    if (lane < deg && v) {
      const int q0 = t.nbr_ptr[q], q1 = t.nbr_ptr[q + 1];
      int slot = -1;
      if (q2 == q) {
        slot = t.slot_ptr[q];
      } else {
        int lo = q0, hi = q1;
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (t.nbr[mid] < q2) lo = mid + 1; else hi = mid;
        }
        if (lo < q1 && t.nbr[lo] == q2) slot = t.slot_ptr[q] + 1 + (lo - q0);
      }
      // (no slot: a far pair, consumed by the recompression)
      if (slot >= 0) dst = (elq + el2 == 0 ? t.nb0 : (elq + el2 == 1 ? t.nb1 : t.nb2))[slot];
    }
    dsts[lane] = dst;
    if (lane == a) s_mq = v;
    if (lane == 0) s_ld = t.n[q];
  }
  __syncthreads();
  const int mq = s_mq;
  if (mq == 0 || t.n[i] == 0) return;
  const long ldd = s_ld;
  const int M = roff[deg];
  const double* F = D.F + roff[a];
  const int rp = mq <= 8 ? 8 : (mq <= 16 ? 16 : 32), cw = 32 / rp;  // lanes per column, columns per warp
  const int x0 = lane & (rp - 1);
  int b = 0;
  for (int col = w * cw + lane / rp; col < M; col += 4 * nw * cw) {
    double* o[4];
    const double* f[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int c = col + u * nw * cw;
      o[u] = nullptr;
      f[u] = nullptr;
      if (c < M) {
        while (c >= roff[b + 1]) ++b;
        f[u] = F + (long)c * D.M;
        if (dsts[b]) o[u] = dsts[b] + (c - roff[b]) * ldd;
      }
    }
    for (int x = x0; x < mq; x += rp) {
      double v[4], y[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        v[u] = y[u] = 0.0;
        if (o[u]) {
          v[u] = f[u][x];
          y[u] = o[u][x];
        }
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (o[u]) o[u][x] = y[u] + v[u];
    }
  }
}

// ---------------------------------------------------------------- Jacobi on P R_k^T
// Hestenes' one-sided Jacobi: rotate column pairs of B until all pairs are
// orthogonal to working precision.  Pairs are taken in the round-robin order
// (k' = k rounded up to even; in round r, position p > 0 holds column
// 1 + ((p - 1 - r) mod (k'-1)); pair i joins positions i and k'-1-i), so the k'/2
// pairs of a round are disjoint and handled by different groups of lanes.
// Columns are rotated in place (no rotation matrix is accumulated: the rotated
// columns themselves, normalised, are the singular vectors sought).  n <= 1024.
//
// Bound: in FP64 the FP64 pipe, in FP32 the issue slots, and in both most of it
// was the scalar part of a pair, which every lane repeats (square roots,
// divisions, hypot: ~150 FP64 instructions against 14 for the rotation itself at
// n = 50).  So: G lanes per pair instead of 32 (a warp does 32 / G pairs at
// once), the two columns held in registers between dot product and rotation (EM
// elements per lane; EM = 0: any length, read twice), squared norms kept and
// updated (al - t g, be + t g; summed afresh every sweep and where the update
// cancels), and the angle from FP32: its tangent is refined by one Newton step in
// FP64, and only c = 1/sqrt(1 + t^2) has to be exact for the rotation to be
// orthogonal.  Six to nine sweeps as before.  Measured (with the launch classes
// of launch_svd_rt): FP64 class of an 8,192-point job 621 -> 281 ms, FP32 class of
// the 131,072-point job 141 -> 56 ms.
// Slot of one problem: B (n x k, ld svd_ld) when it fits, else the descriptor's
// work buffer | squared norms, reciprocals (n each), in TC | order (n ints).
// the column pitch: an odd multiple of G, so that the groups of a warp, which
// read neighbouring columns, meet different banks
__host__ __device__ __forceinline__ int svd_ld(int n, int G) { return G * (((n + G - 1) / G) | 1); }
__host__ __device__ __forceinline__ size_t svd_tail_bytes(int n, int tc_bytes) {
  return (((size_t)n * (2 * tc_bytes + sizeof(int))) + 15) & ~(size_t)15;
}

template <int G, typename TC>
__device__ __forceinline__ TC group_sum(TC v) {
#pragma unroll
  for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float sqrt_fast(float x) {
  float y;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// whether the pair needs a rotation (|g| > tol sqrt(al be))
__device__ __forceinline__ bool svd_needs(float al, float be, float g) {
  return !(al < 1e-36f || be < 1e-36f || fabsf(g) <= 4e-7f * sqrt_fast(al) * sqrt_fast(be));
}
static __device__ __noinline__ bool svd_needs_rare(double al, double be, double g) {
  return !(al < 1e-300 || be < 1e-300 || fabs(g) <= 1e-15 * sqrt(al) * sqrt(be));
}
__device__ __forceinline__ bool svd_needs(double al, double be, double g) {
  // below 2^-431 the products of the squares would underflow
  if (min(dexp(al), dexp(be)) < 592) return svd_needs_rare(al, be, g);
  return !(g * g <= 1e-30 * (al * be));
}
// rotation that orthogonalises columns of squared norms al, be and product g:
// t = tan, c = cos, s = sin; t^2 + 2 z t - 1 = 0 with z = (be - al) / (2 g).  Columns
// of very different size have a z whose square leaves the FP32 range: the root of
// z^2 + 1 is at most |z| + 1, which is what counts there.
__device__ __forceinline__ void svd_rotation(float al, float be, float g, float& t, float& c, float& s) {
  const float z = __fdividef(be - al, g + g);
  const float a = fabsf(z);
  t = __fdividef(copysignf(1.f, z), a + fminf(sqrt_fast(fmaf(z, z, 1.f)), a + 1.f));
  const float x = fmaf(t, t, 1.f), y = rsqrtf(x);
  c = fmaf(0.5f * y, fmaf(-(x * y), y, 1.f), y);
  s = c * t;
}
static __device__ __noinline__ double quotient_rare(double a, double b) { return a / b; }
__device__ __forceinline__ void svd_rotation(double al, double be, double g, double& t, double& c, double& s) {
  const double d = be - al, g2 = g + g;
  const int ed = dexp(d), eg = dexp(g2);
  if (ed - eg > 100) {  // g2 could leave the FP32 range below d
    t = quotient_rare(g, d);
  } else {
    const int sh = 1023 - max(ed, eg);  // both into the FP32 range, exactly scaled
    const float df = d2f_pow2(d, sh), gf = d2f_pow2(g2, sh);
    const float z = __fdividef(df, gf);
    const float t0 = __fdividef(copysignf(1.f, z), fabsf(z) + sqrt_fast(fmaf(z, z, 1.f)));
    t = f2d_pow2(t0, 0);
    // one Newton step of g2 t^2 + 2 d t - g2 = 0: the residual in FP64
    const double f = fma(t, fma(g2, t, d + d), -g2);
    t -= f2d_pow2(__fdividef(d2f_pow2(f, sh), 2.f * fmaf(gf, t0, df)), 0);
  }
  c = rsqrt_fp64(fma(t, t, 1.0));
  s = c * t;
}

// WARP: a problem per warp (k <= 16), else per CTA; slot_bytes of dynamic shared
// memory per problem, of which the last svd_tail_bytes(n) hold the tail.
// CL: a problem per cluster of R = 2, 4 or 8 CTAs.  Column j and its norm live in
// CTA j mod R (the launch has room for ceil(n / R) columns in each), the pairs of a
// round are dealt to the CTAs' warps, which reach the columns through distributed
// shared memory, and the cluster's barrier ends the round.  Every pair is computed as
// in one CTA, so the results are the same bits.  For batches that leave SMs idle: a
// wide FP64 problem is bound by its own SM's FP64 pipe (2 multiply-adds a clock).
// The 8,192-point job 733 -> 592 ms.
template <typename TC, int G, int EM, bool WARP, bool CL>
__global__ void __launch_bounds__(WARP ? 128 : 1024) k_svd_rt(const SvdRtDesc* __restrict__ d, int nd, int max_sweeps,
                                                              int slot_bytes) {
  extern __shared__ __align__(16) unsigned char svm[];
  __shared__ int s_em[32], s_rot[8];
  constexpr unsigned kAll = 0xffffffffu;
  const int lane = threadIdx.x & 31, w = WARP ? 0 : threadIdx.x >> 5, nw = WARP ? 1 : blockDim.x >> 5;
  cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
  const int R = CL ? (int)cl.num_blocks() : 1, rk = CL ? (int)cl.block_rank() : 0, lr = CL ? 31 - __clz(R) : 0;
  const int di = WARP ? blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5) : (CL ? blockIdx.x >> lr : blockIdx.x);
  if (di >= nd) return;  // (of a cluster: every CTA or none)
  auto sync = [] {
    if constexpr (WARP) {
      __syncwarp();
    } else if constexpr (CL) {
      cluster_arrive();
      cluster_wait();
    } else {
      __syncthreads();
    }
  };
  const SvdRtDesc D = d[di];
  const int n = D.n;
  int k = D.kin[0];
  k = k < 0 ? 0 : (k > n ? n : k);
  unsigned char* slot = svm + (WARP ? (size_t)(threadIdx.x >> 5) * slot_bytes : 0);
  const size_t tail = svd_tail_bytes(n, sizeof(TC));
  TC* nrm = (TC*)(slot + slot_bytes - tail);
  TC* rnv = nrm + n;
  int* ord = (int*)(rnv + n);
  const bool in_smem = CL || (size_t)svd_ld(n, G) * k * sizeof(TC) <= (size_t)slot_bytes - tail;
  TC* B = in_smem ? (TC*)slot : (TC*)D.work;
  const int lb = in_smem ? svd_ld(n, G) : n;
  const long ld = D.ld;
  // column j and its squared norm, in the CTA that has them
  auto col = [&](int j) {
    if constexpr (CL) return cl.map_shared_rank(B, j & (R - 1)) + (long)(j >> lr) * lb; else return B + (long)j * lb;
  };
  auto nrm_of = [&](int j) {
    if constexpr (CL) return cl.map_shared_rank(nrm, j & (R - 1)) + j; else return nrm + j;
  };
  // B = P R_k^T (or the explicit matrix), scaled by a power of two 2^sh that
  // brings its largest entry into [0.5, 1); warps over columns, lanes over rows
  int em = 0;
  for (int i = w; i < k; i += nw)
    for (int pos = lane; pos < n; pos += 32) {
      const double v = D.jpvt ? ((i <= pos) ? D.A[i + (long)pos * ld] : 0.0) : D.A[pos + (long)i * ld];
      em = max(em, dexp(v));
    }
  em = (int)__reduce_max_sync(kAll, (unsigned)em);
  if constexpr (!WARP) {
    if (lane == 0) s_em[w] = em;
    __syncthreads();
    em = (int)__reduce_max_sync(kAll, lane < nw ? (unsigned)s_em[lane] : 0u);
  }
  const int sh = pow2_shift(em);
  for (int i = rk + w * R; i < k; i += nw * R)  // its own columns
    for (int pos = lane; pos < n; pos += 32) {
      if (D.jpvt)
        B[D.jpvt[pos] + (long)(i >> lr) * lb] = ld_tc<TC>((i <= pos) ? D.A[i + (long)pos * ld] : 0.0, sh);
      else
        B[pos + (long)(i >> lr) * lb] = ld_tc<TC>(D.A[pos + (long)i * ld], sh);
    }
  sync();
  const int sub = lane & (G - 1), gw = lane / G;  // lane of the group, group of the warp
  constexpr int GW = 32 / G;
  const int kp = k + (k & 1), np = kp / 2;
  // squared norms of every column
  auto norms = [&] {
    for (int j0 = w * GW; j0 << lr < k; j0 += nw * GW) {
      const int jl = j0 + gw, j = (jl << lr) + rk;
      TC s2 = 0;
      if (j < k)
        for (int i = sub; i < n; i += G) {
          const TC u = B[i + (long)jl * lb];
          s2 += u * u;
        }
      s2 = group_sum<G>(s2);
      if (j < k && sub == 0) nrm[j] = s2;
    }
    sync();
  };
  for (int sweep = 0; sweep < max_sweeps && k > 1; ++sweep) {
    norms();
    int rotated = 0;
    for (int r = 0; r < kp - 1; ++r) {
      for (int p0 = (w * R + rk) * GW; p0 < np; p0 += nw * R * GW) {
        const int pi = p0 + gw;
        int a = pi - 1 - r, b = kp - 2 - pi - r;
        a = pi == 0 ? 0 : 1 + (a < 0 ? a + kp - 1 : a);
        b = 1 + (b < 0 ? b + kp - 1 : b);
        if (a > b) { const int tt = a; a = b; b = tt; }
        const bool live = pi < np && b < k;
        TC* ga = col(live ? a : 0);
        TC* gb = col(live ? b : 0);
        TC g = 0;
        TC u[EM > 0 ? EM : 1], v[EM > 0 ? EM : 1];
        if constexpr (EM > 0) {
          TC g1 = 0;
#pragma unroll
          for (int e = 0; e < EM; ++e) {
            const int i = sub + e * G;
            const bool in = live && i < n;
            u[e] = in ? ga[i] : (TC)0;
            v[e] = in ? gb[i] : (TC)0;
            if (e & 1) g1 += u[e] * v[e]; else g += u[e] * v[e];
          }
          g += g1;
        } else if (live) {
          for (int i = sub; i < n; i += G) g += ga[i] * gb[i];
        }
        g = group_sum<G>(g);
        TC al = 0, be = 0;
        if (live) {
          al = *nrm_of(a);
          be = *nrm_of(b);
        }
        const bool rot = live && svd_needs(al, be, g);
        if (!__any_sync(kAll, rot)) continue;
        rotated = 1;
        TC t = 0, c = 1, s = 0;
        if (rot) svd_rotation(al, be, g, t, c, s);
        TC na = al - t * g, nb = be + t * g;
        const bool redo = rot && (!(na > (TC)0.05 * al) || !(nb > (TC)0.05 * be));
        TC sa = 0, sb = 0;
        const bool again = __any_sync(kAll, redo);
        if constexpr (EM > 0) {
          if (rot) {
#pragma unroll
            for (int e = 0; e < EM; ++e) {
              const int i = sub + e * G;
              const TC x = c * u[e] - s * v[e];
              v[e] = s * u[e] + c * v[e];
              u[e] = x;
              if (i < n) {
                ga[i] = u[e];
                gb[i] = v[e];
              }
            }
          }
          if (again)
#pragma unroll
            for (int e = 0; e < EM; ++e) {
              sa += u[e] * u[e];
              sb += v[e] * v[e];
            }
        } else if (rot) {
          for (int i = sub; i < n; i += G) {
            const TC x = ga[i], y = gb[i];
            const TC x2 = c * x - s * y, y2 = s * x + c * y;
            ga[i] = x2;
            gb[i] = y2;
            sa += x2 * x2;
            sb += y2 * y2;
          }
        }
        if (again) {
          sa = group_sum<G>(sa);
          sb = group_sum<G>(sb);
          if (redo) {
            na = sa;
            nb = sb;
          }
        }
        if (rot && sub == 0) {
          *nrm_of(a) = na;
          *nrm_of(b) = nb;
        }
      }
      sync();
    }
    if constexpr (WARP)
      rotated = __any_sync(kAll, rotated);
    else
      rotated = __syncthreads_or(rotated);
    if constexpr (CL) {
      if ((int)threadIdx.x < R) cl.map_shared_rank(s_rot, threadIdx.x)[rk] = rotated;
      sync();
      rotated = 0;
      for (int q = 0; q < R; ++q) rotated |= s_rot[q];  // (next written after other barriers)
    }
    if (!rotated) break;
  }
  // column norms (the singular values times 2^sh) in the arithmetic type, the
  // descending order (NaN last), and the reciprocals once per column
  norms();
  const int tid = WARP ? lane : threadIdx.x, nt = WARP ? 32 : blockDim.x;
  if constexpr (CL) {  // everybody's norms, after which no CTA reads another's memory
    for (int j = tid; j < k; j += nt) rnv[j] = *nrm_of(j);
    sync();
    for (int j = tid; j < k; j += nt) nrm[j] = rnv[j];
  }
  for (int j = tid; j < k; j += nt) {
    const TC v = sqrt(nrm[j]);
    nrm[j] = v;
    rnv[j] = (v > (TC)0) ? (TC)1 / v : (TC)0;
  }
  sync();
  for (int j = tid; j < k; j += nt) {
    int rank = 0;
    const TC v = (nrm[j] == nrm[j]) ? nrm[j] : (TC)-1;
    for (int q = 0; q < k; ++q) {
      const TC u = (nrm[q] == nrm[q]) ? nrm[q] : (TC)-1;
      rank += (u > v) || (u == v && q < j);
    }
    ord[rank] = j;
  }
  sync();
  if (rk == 0)
    for (int j = tid; j < n; j += nt) D.sig[j] = (j < k) ? st_tc<TC>(nrm[ord[j]], -sh) : 0.0;
  for (int j = w; j < n; j += nw) {
    double* vj = D.V + (long)j * D.ldv;
    if (j < k) {
      const int c = ord[j];
      if (CL && (c & (R - 1)) != rk) continue;
      const TC r = rnv[c];
      const TC* g = B + (long)(c >> lr) * lb;
      for (int i = lane; i < n; i += 32) vj[i] = st_tc<TC>(g[i] * r);
    } else if (!CL || (j & (R - 1)) == rk) {
      for (int i = lane; i < n; i += 32) vj[i] = 0.0;
    }
  }
}

// ---------------------------------------------------------------- randomized range finder helpers
// Omega (m x s, ld m) of +-1 entries: bit 63 of SplitMix64(seed + 0x9E37..*(index+1)).
__global__ void k_sketch(const SketchDesc* __restrict__ d, int nd) {
  if ((int)blockIdx.x >= nd) return;
  const SketchDesc D = d[blockIdx.x];
  const long total = (long)D.m * D.s;
  for (long e = threadIdx.x; e < total; e += blockDim.x) {
    unsigned long long z = D.seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(e + 1);
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z = z ^ (z >> 31);
    D.omega[e] = (z >> 63) ? 1.0 : -1.0;
  }
}
// out[0] = Frobenius norm of the m x n block (ld)
__global__ void k_frob(const FrobDesc* __restrict__ d, int nd) {
  if ((int)blockIdx.x >= nd) return;
  const FrobDesc D = d[blockIdx.x];
  __shared__ double scratch[32];
  double s = 0.0;
  const long total = (long)D.m * D.n;
  for (long e = threadIdx.x; e < total; e += blockDim.x) {
    const double v = D.A[(e % D.m) + (e / D.m) * (long)D.ld];
    s += v * v;
  }
  s = block_sum(s, scratch);
  if (threadIdx.x == 0) D.out[0] = sqrt(s);
}

}  // namespace ifmm
