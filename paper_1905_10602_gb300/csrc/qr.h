// Shapes of the register-resident QR (qr.cuh) and its launchers, one translation
// unit per arithmetic type and kind (qr_f32_piv.cu and so on).
#pragma once

#include <cuda_runtime.h>

#include "descs.h"

namespace ifmm {

// rows per lane of the classes of the cluster kernel: class c holds blocks of at
// most 32 kQrRows[c] rows
constexpr int kQrClasses = 8;
constexpr int kQrRows[kQrClasses] = {4, 8, 12, 16, 20, 24, 32, 48};
// columns per lane for E rows per lane, such that the block and the rest stay
// within the 128 registers of a 512-thread CTA
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int qr_class_cols(int E, int tc_bytes) {
  return tc_bytes == 4 ? (E <= 8 ? 8 : (E <= 20 ? 4 : 2)) : (E <= 4 ? 8 : (E <= 12 ? 4 : (E <= 24 ? 2 : 1)));
}
constexpr int kQrMaxWarps = 256;  // of a cluster: 16 CTAs of 16
// the warp-per-problem kernel: at most 16 columns, 64 or 128 rows
constexpr int kQrWarpCols = 16;

// dynamic shared memory of one problem in one CTA: two reflector buffers (32 E
// each, TC) | the warps' keys and columns | pivots, places (n ints each)
#ifdef __CUDACC__
__host__ __device__
#endif
inline size_t qr_reg_bytes(int E, int n, int warps, int tc_bytes) {
  return (((size_t)32 * E * tc_bytes * 2 + (size_t)warps * 12 + 8 * (size_t)n + 16) + 15) & ~(size_t)15;
}

// nd problems of class cls, a cluster of R CTAs of `warps` warps each per problem;
// probe: whether such a cluster can be resident (nothing is launched).  False: not
// launched (or not resident).
bool qr_launch_f32_piv(int cls, const QrcpDesc* d, int nd, int R, int warps, size_t smem, cudaStream_t s, bool probe);
bool qr_launch_f32_plain(int cls, const QrcpDesc* d, int nd, int R, int warps, size_t smem, cudaStream_t s, bool probe);
bool qr_launch_f64_piv(int cls, const QrcpDesc* d, int nd, int R, int warps, size_t smem, cudaStream_t s, bool probe);
bool qr_launch_f64_plain(int cls, const QrcpDesc* d, int nd, int R, int warps, size_t smem, cudaStream_t s, bool probe);
// a warp per problem; tall: up to 128 rows, else 64
void qr_launch_warp_f32_piv(bool tall, const QrcpDesc* d, int nd, cudaStream_t s);
void qr_launch_warp_f32_plain(bool tall, const QrcpDesc* d, int nd, cudaStream_t s);
void qr_launch_warp_f64_piv(bool tall, const QrcpDesc* d, int nd, cudaStream_t s);
void qr_launch_warp_f64_plain(bool tall, const QrcpDesc* d, int nd, cudaStream_t s);

}  // namespace ifmm
