// Householder QR, plain (PIV = false) or with column pivoting stopped at tau_rel,
// of batches of small blocks, each block resident in registers.
//
// A block's columns are dealt cyclically to the warps of one thread-block cluster
// (1 to 16 CTAs; column j to warp j mod W), a lane holding rows lane, lane + 32,
// ...: E rows by C columns per lane.  Only the reflector of a step crosses warps:
// its owner forms v (v_k = 1, v_i = x_i / (x_k - alpha)) from its registers and
// writes it to every CTA's shared memory; every other warp then needs two passes
// over its own registers and one joint reduction of its C dot products.  Columns
// are never moved: a column remembers the step that took it and is written to
// that place at the end.  With pivoting a step has two barriers (the warps' best
// remaining norms; the reflector), without it one: the owner of the next column
// updates that column first and publishes its reflector while the others finish.
//
// Bound: the chain of steps (barriers, one reduction, one square root and one
// reciprocal), then the FP32 issue slots, in FP64 the FP64 pipe -- so what is the
// same for a whole step is computed by one warp, and the joint reduction of C
// columns takes C - 1 + 5 - log2 C additions instead of 5 C.  The shared-memory
// kernels this replaces read every element three times and wrote it once per
// step, and every warp repeated the serial sums, the square root and the
// divisions: QR class of the 131,072-point job (FP32) 286 ms -> 245, of a
// 20,011-point one 96 -> 64, of an 8,192-point FP64 job 420 -> 190, of a
// 2,048-point one 192 -> 55.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "devmath.cuh"
#include "fp64_ops.cuh"
#include "per_device.h"
#include "qr.h"

namespace ifmm {

// An element of the block between its conversions: the FP64 slot, or its first half
// when the arithmetic is FP32.  The conversions are long integer sequences, so they
// stand in two short loops (in, out) over the block in global memory, and the
// unrolled code that fills and empties the registers only moves slots: with the
// conversions unrolled into it the kernels were 200 to 600 KB of code and bound by
// instruction fetch.
// (memcpy: the two types share the storage)
template <typename TC>
__device__ __forceinline__ TC qr_get(const double* p) {
  TC v;
  memcpy(&v, __builtin_assume_aligned(p, 8), sizeof(TC));
  return v;
}
template <typename TC>
__device__ __forceinline__ void qr_put(double* p, TC v) {
  memcpy(__builtin_assume_aligned(p, 8), &v, sizeof(TC));
}
template <typename TC>
__device__ __forceinline__ TC qr_in(double d, int sh) {
  if constexpr (sizeof(TC) == 4) return d2f_pow2(d, sh); else return scale_pow2(d, sh);
}
template <typename TC>
__device__ __forceinline__ double qr_out(TC v, int sh) {
  if constexpr (sizeof(TC) == 4) return f2d_pow2(v, sh); else return scale_pow2(v, sh);
}

// a[c] = sum over the warp of a[c], for all C (a power of two) at once: the
// halves of the list are exchanged between lanes, so that every level adds half
// as many values; every lane gets every sum
template <int C, typename TC>
__device__ __forceinline__ void warp_sums(TC (&a)[C], int lane) {
  int off = 16;
#pragma unroll
  for (int h = C / 2; h >= 1; h >>= 1, off >>= 1) {
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < h; ++i) {
      const TC send = up ? a[i] : a[i + h];
      const TC keep = up ? a[i + h] : a[i];
      a[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  for (; off >= 1; off >>= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], off);
  const TC s = a[0];
#pragma unroll
  for (int c = 0; c < C; ++c) {
    int src = 0;
    for (int h = C / 2, o = 16; h >= 1; h >>= 1, o >>= 1) src |= (c & h) ? o : 0;
    a[c] = __shfl_sync(0xffffffffu, s, src);
  }
}

// alpha, tau and 1 / (x0 - alpha) of the reflector of a column with leading entry
// x0 and squared norm ss below it; tau = 0 where nothing is below
__device__ __forceinline__ void reflector(float x0, float ss, float& alpha, float& tau, float& sc) {
  alpha = x0;
  tau = sc = 0.f;
  const float nr = sqrtf(fmaf(x0, x0, ss));
  if (nr == 0.f || ss == 0.f) return;
  alpha = x0 >= 0.f ? -nr : nr;
  tau = (alpha - x0) / alpha;
  sc = 1.f / (x0 - alpha);
}
__device__ __forceinline__ void reflector(double x0, double ss, double& alpha, double& tau, double& sc) {
  alpha = x0;
  tau = sc = 0.0;
  const double s2 = fma(x0, x0, ss);
  if (s2 == 0.0 || ss == 0.0) return;
  const double rs = rsqrt_fp64(s2), nr = s2 * rs;
  alpha = x0 >= 0.0 ? -nr : nr;
  tau = fma(fabs(x0), rs, 1.0);
  sc = rcp_fp64(x0 - alpha);
}
// order-preserving key of a squared norm (anything not positive: 0)
__device__ __forceinline__ unsigned long long norm_key(float v) {
  return v > 0.f ? (unsigned long long)__float_as_uint(v) << 32 : 0ull;
}
__device__ __forceinline__ unsigned long long norm_key(double v) {
  return v > 0.0 ? (unsigned long long)__double_as_longlong(v) : 0ull;
}
template <typename TC>
__device__ __forceinline__ TC key_norm(unsigned hi, unsigned lo) {
  if constexpr (sizeof(TC) == 4) return __uint_as_float(hi); else return __hiloint2double((int)hi, (int)lo);
}

// p ? a : b on values (a conditional on array elements may select addresses, and an
// array whose address is taken leaves the registers)
template <typename TC>
__device__ __forceinline__ TC pick(bool p, TC a, TC b) { return p ? a : b; }

// the reflector of column c0 with its leading entry in lane kl of e = 0: the lane's
// entries to v[32 e], the column becomes R's; returns tau
template <typename TC, int E, int C, class P>
__device__ __forceinline__ TC qr_reflect(TC (&y)[C][E], int c0, int kl, int lane, P&& put_v) {
  auto x = [&](int e) __attribute__((always_inline)) {
    TC q = y[0][e];
#pragma unroll
    for (int c = 1; c < C; ++c) q = pick<TC>(c == c0, y[c][e], q);
    return q;
  };
  const TC y0 = x(0);
  const TC x0 = __shfl_sync(0xffffffffu, y0, kl);
  TC ss = pick<TC>(lane > kl, y0 * y0, (TC)0), s1 = 0;
#pragma unroll
  for (int e = 1; e < E; ++e) {
    const TC q = x(e);
    if (e & 1) s1 += q * q; else ss += q * q;
  }
  ss = warp_sum_t<TC>(ss + s1);
  TC alpha, tau, sc;
  reflector(x0, ss, alpha, tau, sc);
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const TC xe = x(e);
    TC z = 0, v = sc * xe;
    if (e == 0) {
      z = pick<TC>(lane > kl, (TC)0, pick<TC>(lane == kl, alpha, xe));
      v = pick<TC>(lane > kl, v, (TC)(lane == kl));
    }
    put_v(e, v);
#pragma unroll
    for (int c = 0; c < C; ++c) y[c][e] = pick<TC>(c == c0, z, y[c][e]);
  }
  return tau;
}
// the columns with on[c] -= tau v (v . y)
template <typename TC, int E, int C>
__device__ __forceinline__ void qr_apply(TC (&y)[C][E], const bool (&on)[C], const TC* vb, TC tau, int lane) {
  const TC* v = vb + lane;
  TC a[C];
#pragma unroll
  for (int c = 0; c < C; ++c) a[c] = 0;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const TC ve = v[e * 32];
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (on[c]) a[c] += ve * y[c][e];
  }
  warp_sums<C>(a, lane);
#pragma unroll
  for (int c = 0; c < C; ++c) a[c] *= -tau;
#pragma unroll
  for (int e = 0; e < E; ++e) {
    const TC ve = v[e * 32];
#pragma unroll
    for (int c = 0; c < C; ++c)
      if (on[c]) y[c][e] += a[c] * ve;
  }
}

// WARP: one warp per problem (n <= C, m <= 32 E), several per CTA; else a cluster
// per problem (n <= C * warps of the cluster)
template <typename TC, int E, int C, bool PIV, bool WARP>
__global__ void __launch_bounds__(WARP ? 128 : 512, 1) k_qr_reg(const QrcpDesc* __restrict__ d, int nd, int slot) {
  namespace cg = cooperative_groups;
  constexpr unsigned kAll = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char qsm[];
  __shared__ int xe[WARP ? 1 : kQrMaxWarps];  // largest exponent per warp of the cluster
  __shared__ TC s_tau[2];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  cg::cluster_group cl = cg::this_cluster();
  const int R = WARP ? 1 : (int)cl.num_blocks(), rank = WARP ? 0 : (int)cl.block_rank();
  const int nw = WARP ? 1 : (int)(blockDim.x >> 5), W = R * nw;
  const int gw = WARP ? 0 : rank * nw + wp;
  const int pi = WARP ? blockIdx.x * (blockDim.x >> 5) + wp : blockIdx.x / R;
  if (WARP && pi >= nd) return;
  const QrcpDesc D = d[pi < nd ? pi : nd - 1];
  const int m = D.m, n = D.n;
  const long ld = D.ld;
  unsigned char* sl = qsm + (WARP ? (size_t)wp * slot : 0);
  TC* vb = (TC*)sl;  // two buffers of 32 E
  unsigned long long* kv = (unsigned long long*)(vb + 2 * 32 * E);
  int* ki = (int*)(kv + W);
  int* pv = ki + W;    // column of step s
  int* place = pv + n; // place of column j
  auto bar = [&] {
    if constexpr (WARP) {
      __syncwarp();
    } else if (R == 1) {
      __syncthreads();
    } else {
      cluster_arrive();
      cluster_wait();
    }
  };
  // p in CTA r's shared memory
  auto at = [&](auto* p, int r) {
    if constexpr (WARP) return p; else return R == 1 ? p : cl.map_shared_rank(p, r);
  };
  // power-of-two scale that brings the largest magnitude into [0.5, 1)
  int em = 0;
#pragma unroll 1
  for (int j = gw; j < n; j += W) {
    const double* col = D.A + (long)j * ld;
    if (D.rb > 0) {
#pragma unroll 1
      for (int i = lane; i < m; i += 32) em = max(em, dexp(col[qr_row(D, i)]));
    } else {
#pragma unroll 8
      for (int i = lane; i < m; i += 32) em = max(em, dexp(col[i]));
    }
  }
  em = (int)__reduce_max_sync(kAll, (unsigned)em);
  if constexpr (!WARP) {
    if (R > 1) bar();  // every CTA runs before another writes into it
    if (lane == 0) {
#pragma unroll 1
      for (int r = 0; r < R; ++r) at(xe, r)[gw] = em;
    }
    bar();
    em = 0;
#pragma unroll 1
    for (int x = lane; x < W; x += 32) em = max(em, xe[x]);
    em = (int)__reduce_max_sync(kAll, (unsigned)em);
  }
  const int sh = pow2_shift(em);
  // into slots; stacked rows (rb > 0) move up to their logical places (a row's
  // place is never below what is still to be read of its column)
#pragma unroll 1
  for (int j = gw; j < n; j += W) {
    double* col = D.A + (long)j * ld;
    if (D.rb > 0) {
#pragma unroll 1
      for (int i0 = 0; i0 < m; i0 += 32) {
        const int i = i0 + lane;
        const double v = i < m ? col[qr_row(D, i)] : 0.0;
        __syncwarp();
        if (i < m) qr_put<TC>(col + i, qr_in<TC>(v, sh));
        __syncwarp();
      }
    } else {
#pragma unroll 4
      for (int i = lane; i < m; i += 32) qr_put<TC>(col + i, qr_in<TC>(col[i], sh));
    }
  }
  TC y[C][E];
  bool live[C];  // a column of the block, not yet taken by a step
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const int j = gw + c * W;
    live[c] = j < n;
    const double* col = D.A + (long)j * ld + lane;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      y[c][e] = 0;
      if (j < n && e * 32 + lane < m) y[c][e] = qr_get<TC>(col + e * 32);
    }
  }
  const int kmax = m < n ? m : n;
  // Step k's row is always in e = 0: after every 32 steps the 32 finished rows go
  // to this warp's own columns of A (all of which is in registers) and the rest
  // moves up.
  int done = 0;  // blocks of 32 rows that have gone
  auto shift = [&] {
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const int j = gw + c * W, i = 32 * done + lane;
      if (j < n && i < kmax) qr_put<TC>(D.A + i + (long)j * ld, y[c][0]);
#pragma unroll
      for (int e = 0; e + 1 < E; ++e) y[c][e] = y[c][e + 1];
      y[c][E - 1] = 0;
    }
    ++done;
  };
  // the reflector of step k from this warp's column c0, to every CTA's buffer b
  auto publish = [&](int c0, int k, int b) __attribute__((always_inline)) {
    TC* v0 = vb + b * 32 * E + lane;
    const TC tau =
        qr_reflect<TC, E, C>(y, c0, k & 31, lane, [&](int e, TC v) __attribute__((always_inline)) { v0[e * 32] = v; });
    if constexpr (!WARP) {
#pragma unroll 1
      for (int r = 0; r < R; ++r) {
        if (r == rank) continue;
        TC* v1 = cl.map_shared_rank(v0, r);
#pragma unroll
        for (int e = 0; e < E; ++e) v1[e * 32] = v0[e * 32];
      }
    }
#pragma unroll
    for (int c = 0; c < C; ++c) live[c] = live[c] && c != c0;
    if (lane == 0) {
      if constexpr (WARP) {
        vb[64 * E - 1] = tau;  // the second buffer, which a single warp does not use
      } else {
#pragma unroll 1
        for (int r = 0; r < R; ++r) at(s_tau, r)[b] = tau;
      }
    }
  };
  auto tau_of = [&](int b) {
    if constexpr (WARP) return vb[64 * E - 1]; else return s_tau[b];
  };
  int k = 0;
  bool capped = false;
  double tailv = 0.0;
  if constexpr (PIV) {
    TC nrm[C], ref[C];
#pragma unroll
    for (int c = 0; c < C; ++c) {
      TC s = 0;
#pragma unroll
      for (int e = 0; e < E; ++e) s += y[c][e] * y[c][e];
      nrm[c] = s;
    }
    warp_sums<C>(nrm, lane);
#pragma unroll
    for (int c = 0; c < C; ++c) ref[c] = nrm[c];
    TC tau2 = 0, first = 0;
#pragma unroll 1
    for (; k < kmax; ++k) {
      // this warp's best remaining column (ties: smallest), then everybody's
      unsigned long long bk = 0;
      int bj = 0x7fffffff;
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const unsigned long long q = live[c] ? norm_key(nrm[c]) : 0ull;
        if (live[c] && (bj == 0x7fffffff || q > bk)) {
          bk = q;
          bj = gw + c * W;
        }
      }
      unsigned hi = (unsigned)(bk >> 32), lo = (unsigned)bk;
      int p = bj;
      if constexpr (!WARP) {
        if (lane == 0) {
#pragma unroll 1
          for (int r = 0; r < R; ++r) {
            at(kv, r)[gw] = bk;
            at(ki, r)[gw] = bj;
          }
        }
        bar();
        hi = lo = 0;
        p = 0x7fffffff;
#pragma unroll 1
        for (int x = lane; x < W; x += 32) {
          const unsigned h = (unsigned)(kv[x] >> 32), l = (unsigned)kv[x];
          const int j = ki[x];
          if (h > hi || (h == hi && (l > lo || (l == lo && j < p)))) {
            hi = h;
            lo = l;
            p = j;
          }
        }
        warp_max_key(hi, lo, p);
      }
      const TC best = key_norm<TC>(hi, lo);
      if (k == 0) {
        tau2 = (TC)(D.tau_rel * D.tau_rel) * best;
        first = best;
      }
      bool stop = !(best > tau2) || !(best > (TC)0) || p >= n;
      if (!stop && D.kcap > 0 && k >= D.kcap) {
        stop = true;
        capped = true;
        tailv = (first > (TC)0) ? sqrt((double)best / (double)first) : 0.0;
      }
      if (stop) break;
      if ((WARP ? lane : (int)threadIdx.x) == 0) pv[k] = p;
      if (p % W == gw) publish(p / W, k, 0);
      bar();
      const TC tau = tau_of(0);
      if (tau != (TC)0) qr_apply<TC, E, C>(y, live, vb, tau, lane);
      // downdate the norms with row k; summed afresh where two digits have gone
      bool low = false;
      TC nv[C];
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const TC r = __shfl_sync(kAll, y[c][0], k & 31);
        nv[c] = nrm[c] - r * r;
        low = low || (live[c] && !(nv[c] > (TC)1e-2 * ref[c]));
      }
      if (low) {  // the same in every lane
        TC s[C];
#pragma unroll
        for (int c = 0; c < C; ++c) {
          s[c] = pick<TC>(lane > (k & 31), y[c][0] * y[c][0], (TC)0);
#pragma unroll
          for (int e = 1; e < E; ++e) s[c] += y[c][e] * y[c][e];
        }
        warp_sums<C>(s, lane);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          const bool again = !(nv[c] > (TC)1e-2 * ref[c]);
          nv[c] = pick<TC>(again, s[c], nv[c]);
          ref[c] = pick<TC>(again, s[c], ref[c]);
        }
      }
#pragma unroll
      for (int c = 0; c < C; ++c) nrm[c] = nv[c];
      if ((k & 31) == 31) shift();
      if constexpr (WARP) __syncwarp();  // every lane has read v
    }
  } else {
    // one barrier per step (the reflector buffers alternate)
    if (gw == 0 && kmax > 0) publish(0, 0, 0);
    bar();
#pragma unroll 1
    for (; k < kmax; ++k) {
      const int b = WARP ? 0 : k & 1;
      const TC tau = tau_of(b);
      if (tau != (TC)0) qr_apply<TC, E, C>(y, live, vb + b * 32 * E, tau, lane);
      if ((k & 31) == 31) shift();
      if constexpr (WARP) __syncwarp();  // every lane has read v
      if (k + 1 < kmax && (k + 1) % W == gw) publish((k + 1) / W, k + 1, WARP ? 0 : b ^ 1);
      bar();
    }
  }
  // places: the column of step s at s, the rest behind in index order
  const int tid = WARP ? lane : (int)threadIdx.x, nt = WARP ? 32 : (int)blockDim.x;
  if constexpr (PIV) {
    bar();
#pragma unroll 1
    for (int j = tid; j < n; j += nt) place[j] = -1;
    if constexpr (WARP) __syncwarp(); else __syncthreads();
#pragma unroll 1
    for (int s = tid; s < k; s += nt) place[pv[s]] = s;
    if constexpr (WARP) __syncwarp(); else __syncthreads();
    if (WARP || wp == 0) {
      int next = k;
#pragma unroll 1
      for (int j0 = 0; j0 < n; j0 += 32) {
        const int j = j0 + lane;
        const bool un = j < n && place[j] < 0;
        const unsigned mask = __ballot_sync(kAll, un);
        if (un) place[j] = next + __popc(mask & ((1u << lane) - 1u));
        next += __popc(mask);
      }
    }
    if constexpr (WARP) __syncwarp(); else __syncthreads();
    if (rank == 0) {
#pragma unroll 1
      for (int j = tid; j < n; j += nt) D.jpvt[place[j]] = j;
      if (tid == 0) {
        D.kout[0] = k;
        if (D.tail) D.tail[0] = (k < kmax && capped) ? tailv : 0.0;
      }
    }
  }
  if constexpr (PIV) {
    // take the finished rows back before any column is written to its place
#pragma unroll 1
    for (int q = done - 1; q >= 0; --q)
#pragma unroll
      for (int c = 0; c < C; ++c) {
        const int j = gw + c * W, i = 32 * q + lane;
#pragma unroll
        for (int e = E - 1; e > 0; --e) y[c][e] = y[c][e - 1];
        y[c][0] = 0;
        if (j < n && i < kmax) y[c][0] = qr_get<TC>(D.A + i + (long)j * ld);
      }
    if (done) bar();
    done = 0;
  }
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const int j = gw + c * W;
    if (j >= n) continue;
    double* col = D.A + (long)(PIV ? place[j] : j) * ld + 32 * done + lane;
#pragma unroll
    for (int e = 0; e < E; ++e)
      if ((e + done) * 32 + lane < kmax) qr_put<TC>(col + e * 32, y[c][e]);
  }
  // out of the slots, by the lanes that filled them
#pragma unroll 1
  for (int j = gw; j < n; j += W) {
    double* col = D.A + (long)(PIV ? place[j] : j) * ld;
#pragma unroll 4
    for (int i = lane; i < kmax; i += 32) qr_put<double>(col + i, qr_out<TC>(qr_get<TC>(col + i), -sh));
  }
  if constexpr (!WARP)
    if (R > 1) bar();  // no CTA leaves while another may still write into it
}

// ---------------------------------------------------------------- shapes and launches
template <typename TC, int E, bool PIV>
bool qr_launch_e(const QrcpDesc* d, int nd, int R, int warps, size_t smem, cudaStream_t s, bool probe) {
  auto f = k_qr_reg<TC, E, qr_class_cols(E, sizeof(TC)), PIV, false>;
  static PerDevice<std::once_flag> attr_once;
  std::call_once(attr_once(), [&] {
    if (cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) cudaGetLastError();
  });
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nd * R), 1, 1);
  cfg.blockDim = dim3((unsigned)(32 * warps), 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)R;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (probe) {
    int ncl = 0;
    if (cudaOccupancyMaxActiveClusters(&ncl, f, &cfg) != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    return ncl > 0;
  }
  return cudaLaunchKernelEx(&cfg, f, d, nd, 0) == cudaSuccess;
}
template <typename TC, bool PIV>
bool qr_launch_c(int cls, const QrcpDesc* d, int nd, int R, int warps, size_t smem, cudaStream_t s, bool probe) {
  switch (cls) {
    case 0: return qr_launch_e<TC, 4, PIV>(d, nd, R, warps, smem, s, probe);
    case 1: return qr_launch_e<TC, 8, PIV>(d, nd, R, warps, smem, s, probe);
    case 2: return qr_launch_e<TC, 12, PIV>(d, nd, R, warps, smem, s, probe);
    case 3: return qr_launch_e<TC, 16, PIV>(d, nd, R, warps, smem, s, probe);
    case 4: return qr_launch_e<TC, 20, PIV>(d, nd, R, warps, smem, s, probe);
    case 5: return qr_launch_e<TC, 24, PIV>(d, nd, R, warps, smem, s, probe);
    case 6: return qr_launch_e<TC, 32, PIV>(d, nd, R, warps, smem, s, probe);
    default: return qr_launch_e<TC, 48, PIV>(d, nd, R, warps, smem, s, probe);
  }
}
template <typename TC, bool PIV>
void qr_launch_w(int tall, const QrcpDesc* d, int nd, cudaStream_t s) {
  const unsigned g = (unsigned)((nd + 3) / 4);
  if (tall) {
    const int slot = (int)qr_reg_bytes(4, 16, 1, sizeof(TC));
    k_qr_reg<TC, 4, 16, PIV, true><<<g, 128, 4 * slot, s>>>(d, nd, slot);
  } else {
    const int slot = (int)qr_reg_bytes(2, 16, 1, sizeof(TC));
    k_qr_reg<TC, 2, 16, PIV, true><<<g, 128, 4 * slot, s>>>(d, nd, slot);
  }
}

}  // namespace ifmm
