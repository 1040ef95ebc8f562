// Rank predictor: a small MLP (9 -> 64 -> 64 -> 64 -> 1, ReLU, FP32) that maps
// a recompression event's geometry (cell centre, size, level, offset to the
// eliminated neighbour) and log10(eps) to the truncation rank / 64.  Forward,
// backward and Adam kernels are written here; training runs on the GPU on the
// ranks that the SVD-mode factorization chose.
//
// Weight layout (floats, row-major W[in][out]): W1[9][64] b1[64] W2[64][64] b2[64]
// W3[64][64] b3[64] W4[64][1] b4[1]  -- IFMM_MLP_NWEIGHTS = 9025.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "common.h"
#include "mlp.h"
#include "pairs.cuh"
#include "per_device.h"
#include "runtime.h"

namespace ifmm {

static const int kIn = IFMM_MLP_IN, kH = 64;
static const int kDims[5] = {kIn, kH, kH, kH, 1};

// offsets of W_l and b_l in the flat weight vector
static void layer_offsets(int l, int* w, int* b) {
  int o = 0;
  for (int q = 0; q < l; ++q) o += kDims[q] * kDims[q + 1] + kDims[q + 1];
  *w = o;
  *b = o + kDims[l] * kDims[l + 1];
}

// ---------------------------------------------------------------- the fused pass
// One CTA takes tiles of 64 samples through the whole network with every weight
// and every activation of the tile in shared memory; nothing but the inputs, the
// targets and the results touches global memory.  512 threads, a 4 x 2 patch of
// a 64 x 64 layer each (warp ty: rows ty + 16 u, lane tx: columns tx + 32 v): the
// row operand is a broadcast and the column operand 32 consecutive words, and
// the odd row pitch keeps the transposed reads of the backward pass free of bank
// conflicts as well.  GRAD: the weight gradients stay in registers as float pairs
// across all tiles of the CTA (exact products, two-sums: 10 FP32 operations
// instead of one FP64 multiply-add, which occupies GB300's narrow FP64 pipe for
// 64 FP32 slots), and are written once per CTA; k_mlp_reduce adds the CTAs'
// parts in FP64 in CTA order.  A CTA whose factors are too large or too small for
// exact products in FP32's range (mlp_fits) does its tiles again with FP64 sums.
// Bound by the FP32 issue rate of the pair sums.
// 65,536 rows, one forward and one gradient call with their host copies: 0.83 ms,
// against 75 ms for a kernel per layer whose weight gradient was one thread per
// weight walking every row in FP64 (36 CTAs).
constexpr int kT = 64, kP = 65;  // samples of a tile; row pitch of 64-wide matrices
constexpr int kMlpThreads = 512;
// shared memory (floats): W2, W3 (64 x 65), W1 (9 x 64), b1, b2, b3, W4 (64 each), b4 (4), X (64 x 9), dy (64),
// A1, A2, A3 (64 x 65), then for the gradient G2, G3
constexpr int kSmW2 = 0, kSmW3 = kSmW2 + 64 * kP, kSmW1 = kSmW3 + 64 * kP, kSmB = kSmW1 + 576, kSmX = kSmB + 260,
              kSmDy = kSmX + kT * 9, kSmA = kSmDy + kT, kSmG = kSmA + 3 * kT * kP, kSmEnd = kSmG + 2 * kT * kP;
constexpr int mlp_smem_bytes(bool grad) { return 4 * (grad ? kSmEnd : kSmG); }

__device__ __forceinline__ void mac(df& acc, float a, float b) {
  const float p = a * b;
  const df s = df_two_sum(acc.h, p);
  acc.h = s.h;
  acc.l += s.l + fmaf(a, b, -p);
}
__device__ __forceinline__ void mac(double& acc, float a, float b) { acc = fma((double)a, (double)b, acc); }
__device__ __forceinline__ double sum_of(df v) { return (double)v.h + (double)v.l; }
__device__ __forceinline__ double sum_of(double v) { return v; }

// Smallest nonzero (less one, so that zeros do not count) and largest magnitude of a
// set of floats, as bits.
struct MlpRange {
  unsigned lo = 0xffffffffu, hi = 0u;
  __device__ __forceinline__ void add(float v) {
    const unsigned u = __float_as_uint(v) & 0x7fffffffu;
    lo = min(lo, u - 1u);
    hi = max(hi, u);
  }
};
// Whether the factors a in A (and 1) and g in G of the CTA's threads can be multiplied
// and summed as float pairs like FP64 would: finite, the last bit of every product a
// multiple of 2^-149 (exponents from -103 on), and sums of 2^20 products below 2^127
// (a CTA has at most 2^26 / 152 + 64 samples).  Every thread gets the answer.
__device__ __forceinline__ bool mlp_fits(MlpRange A, MlpRange G) {
  __shared__ unsigned r[4];
  constexpr unsigned kAll = 0xffffffffu;
  if (threadIdx.x < 4) r[threadIdx.x] = threadIdx.x & 1 ? 0u : kAll;
  __syncthreads();
  const unsigned v[4] = {__reduce_min_sync(kAll, A.lo), __reduce_max_sync(kAll, A.hi), __reduce_min_sync(kAll, G.lo),
                         __reduce_max_sync(kAll, G.hi)};
  if ((threadIdx.x & 31) == 0) {
    atomicMin(r, v[0]);
    atomicMax(r + 1, v[1]);
    atomicMin(r + 2, v[2]);
    atomicMax(r + 3, v[3]);
  }
  __syncthreads();
  const unsigned ah = r[1], gh = r[3];
  if (max(ah, gh) >= 0x7f800000u) return false;
  if (gh == 0u) return true;
  const int la = (int)((r[0] + 1u) >> 23) - 127, lg = (int)((r[2] + 1u) >> 23) - 127;
  return (ah == 0u || la + lg >= -103) && max((int)(ah >> 23) - 127, 0) + (int)(gh >> 23) - 127 <= 105;
}

// C[s][j] = relu(b[j] + sum_i A[s][i] W[i][j]), i ascending; zero from sample cnt on
// (a sample that is not there adds exact zeros to the gradient, whatever the weights)
__device__ __forceinline__ void mlp_hidden(const float* A, const float* W, const float* b, float* C, int cnt, int tx,
                                           int ty, MlpRange& rg) {
  float acc[4][2];
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) acc[u][v] = b[tx + 32 * v];
#pragma unroll 8
  for (int i = 0; i < 64; ++i) {
    float w[2], x[4];
#pragma unroll
    for (int v = 0; v < 2; ++v) w[v] = W[i * kP + tx + 32 * v];
#pragma unroll
    for (int u = 0; u < 4; ++u) x[u] = A[(ty + 16 * u) * kP + i];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) acc[u][v] = fmaf(x[u], w[v], acc[u][v]);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const float r = ty + 16 * u < cnt ? fmaxf(acc[u][v], 0.f) : 0.f;
      C[(ty + 16 * u) * kP + tx + 32 * v] = r;
      rg.add(r);
    }
}
// D[s][i] = (sum_j G[s][j] W[i][j]) relu'(A[s][i]), j ascending
__device__ __forceinline__ void mlp_back(const float* G, const float* W, const float* A, float* D, int tx, int ty,
                                         MlpRange& rg) {
  float acc[4][2] = {};
#pragma unroll 8
  for (int j = 0; j < 64; ++j) {
    float w[2], g[4];
#pragma unroll
    for (int v = 0; v < 2; ++v) w[v] = W[(tx + 32 * v) * kP + j];
#pragma unroll
    for (int u = 0; u < 4; ++u) g[u] = G[(ty + 16 * u) * kP + j];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) acc[u][v] = fmaf(g[u], w[v], acc[u][v]);
  }
#pragma unroll
  for (int u = 0; u < 4; ++u)
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const int e = (ty + 16 * u) * kP + tx + 32 * v;
      const float r = A[e] > 0.f ? acc[u][v] : 0.f;
      D[e] = r;
      rg.add(r);
    }
}
// acc[u][v] += sum_s A[s][ty + 16 u] G[s][tx + 32 v]
template <class ACC>
__device__ __forceinline__ void mlp_outer(const float* A, const float* G, ACC (&acc)[4][2], int tx, int ty) {
#pragma unroll 2
  for (int s = 0; s < kT; ++s) {
    float a[4], g[2];
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] = A[s * kP + ty + 16 * u];
#pragma unroll
    for (int v = 0; v < 2; ++v) g[v] = G[s * kP + tx + 32 * v];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) mac(acc[u][v], a[u], g[v]);
  }
}

// The CTA's tiles, weights staged (a barrier follows here): y[s] (may be NULL with GRAD)
// for samples s < ns; GRAD: o[IFMM_MLP_NWEIGHTS + 1] = the CTA's sums of the gradient
// of L = mean (y - t)^2 / 2, kept as ACC, and, last, of the samples' (y - t)^2 / 2.
// Returns, in every thread, whether float pairs hold the sums (mlp_fits).
template <bool GRAD, class ACC>
__device__ __forceinline__ bool mlp_tiles(float* sm, const float* __restrict__ x, const float* __restrict__ t,
                                          float* __restrict__ y, double* __restrict__ o, int ns) {
  float *W2 = sm + kSmW2, *W3 = sm + kSmW3, *W1 = sm + kSmW1, *B = sm + kSmB, *X = sm + kSmX, *dy = sm + kSmDy;
  float *A1 = sm + kSmA, *A2 = A1 + kT * kP, *A3 = A2 + kT * kP, *G2 = sm + kSmG, *G3 = G2 + kT * kP;
  const int tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  ACC w2[4][2] = {}, w3[4][2] = {}, w1[2] = {}, wb = {};
  MlpRange ra, rg;
  double sq = 0.0;
  const int ntile = (ns + kT - 1) / kT;
  for (int tile = blockIdx.x; tile < ntile; tile += gridDim.x) {
    const int s0 = tile * kT, cnt = min(kT, ns - s0);
    __syncthreads();  // weights staged; the previous tile is done with X and dy
    for (int e = tid; e < kT * 9; e += kMlpThreads) {
      const float v = e < cnt * 9 ? x[(long)s0 * 9 + e] : 0.f;
      X[e] = v;
      ra.add(v);
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int s = ty + 16 * u, j = tx + 32 * v;
        float acc = B[j];
#pragma unroll
        for (int i = 0; i < 9; ++i) acc = fmaf(X[s * 9 + i], W1[i * 64 + j], acc);
        acc = s < cnt ? fmaxf(acc, 0.f) : 0.f;
        A1[s * kP + j] = acc;
        ra.add(acc);
      }
    __syncthreads();
    mlp_hidden(A1, W2, B + 64, A2, cnt, tx, ty, ra);
    __syncthreads();
    mlp_hidden(A2, W3, B + 128, A3, cnt, tx, ty, ra);
    __syncthreads();
    if (tid < kT) {
      float acc = B[256];
#pragma unroll 8
      for (int i = 0; i < 64; ++i) acc = fmaf(A3[tid * kP + i], B[192 + i], acc);
      if (y && tid < cnt) y[s0 + tid] = acc;
      if (GRAD) {
        const float d = tid < cnt ? acc - t[s0 + tid] : 0.f;
        const float dn = d / (float)ns;
        dy[tid] = dn;
        rg.add(dn);
        sq += (double)(0.5f * d * d);
      }
    }
    if constexpr (GRAD) {
      __syncthreads();
      // gradient of the last hidden layer; W4 and the biases: thread tid < 64 sums W4[tid], then 65 and on the biases
#pragma unroll
      for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          const int e = (ty + 16 * u) * kP + tx + 32 * v;
          const float g = fmaf(dy[ty + 16 * u], B[192 + tx + 32 * v], 0.f);
          const float r = A3[e] > 0.f ? g : 0.f;
          G3[e] = r;
          rg.add(r);
        }
      __syncthreads();
      mlp_back(G3, W3, A2, G2, tx, ty, rg);
      mlp_outer(A2, G3, w3, tx, ty);
      if (tid < 64) {
        for (int s = 0; s < kT; ++s) mac(wb, A3[s * kP + tid], dy[s]);
      } else if (tid < 128) {
        for (int s = 0; s < kT; ++s) mac(wb, G3[s * kP + tid - 64], 1.f);
      } else if (tid == 128) {
        for (int s = 0; s < kT; ++s) mac(wb, dy[s], 1.f);
      }
      __syncthreads();
      mlp_outer(A1, G2, w2, tx, ty);
      if (tid >= 160 && tid < 224)
        for (int s = 0; s < kT; ++s) mac(wb, G2[s * kP + tid - 160], 1.f);
      __syncthreads();
      mlp_back(G2, W2, A1, G3, tx, ty, rg);  // G3 now holds the gradient of the first hidden layer
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int e = tid + q * kMlpThreads;
        if (e < 576)
          for (int s = 0; s < kT; ++s) mac(w1[q], X[s * 9 + (e >> 6)], G3[s * kP + (e & 63)]);
      }
      if (tid >= 256 && tid < 320)
        for (int s = 0; s < kT; ++s) mac(wb, G3[s * kP + tid - 256], 1.f);
    }
  }
  if constexpr (GRAD) {
    auto put = [&](int e, ACC v) { o[e] = sum_of(v); };
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const int e = (ty + 16 * u) * 64 + tx + 32 * v;
        put(640 + e, w2[u][v]);
        put(4800 + e, w3[u][v]);
      }
    put(tid, w1[0]);
    if (tid < 64) put(512 + tid, w1[1]);
    if (tid < 64) put(8960 + tid, wb);                          // W4
    if (tid >= 64 && tid < 128) put(8896 + tid - 64, wb);       // b3
    if (tid == 128) put(9024, wb);                              // b4
    if (tid >= 160 && tid < 224) put(4736 + tid - 160, wb);     // b2
    if (tid >= 256 && tid < 320) put(576 + tid - 256, wb);      // b1
    __syncthreads();
    double* sqs = (double*)(sm + kSmA);  // 8-byte aligned: kSmA is even
    if (tid < kT) sqs[tid] = sq;
    __syncthreads();
    if (tid == 0) {
      double a = 0.0;
      for (int i = 0; i < kT; ++i) a += sqs[i];
      o[IFMM_MLP_NWEIGHTS] = a;
    }
  }
  if constexpr (GRAD && std::is_same<ACC, df>::value)
    return mlp_fits(ra, rg);
  else
    return true;
}

template <bool GRAD>
__global__ void __launch_bounds__(kMlpThreads) k_mlp(const float* __restrict__ w, const float* __restrict__ x,
                                                     const float* __restrict__ t, float* __restrict__ y,
                                                     double* __restrict__ part, int ns) {
  extern __shared__ float sm[];
  float *W2 = sm + kSmW2, *W3 = sm + kSmW3, *W1 = sm + kSmW1, *B = sm + kSmB;
  const int tid = threadIdx.x;
  for (int e = tid; e < 576; e += kMlpThreads) W1[e] = w[e];
  for (int e = tid; e < 4096; e += kMlpThreads) {
    W2[(e >> 6) * kP + (e & 63)] = w[640 + e];
    W3[(e >> 6) * kP + (e & 63)] = w[4800 + e];
  }
  for (int e = tid; e < 64; e += kMlpThreads) {
    B[e] = w[576 + e];
    B[64 + e] = w[4736 + e];
    B[128 + e] = w[8896 + e];
    B[192 + e] = w[8960 + e];
  }
  if (tid == 0) B[256] = w[9024];
  if constexpr (GRAD) {
    double* o = part + (long)blockIdx.x * (IFMM_MLP_NWEIGHTS + 1);
    // where a factor is too large or too small for pairs, all over again in FP64
    if (!mlp_tiles<true, df>(sm, x, t, y, o, ns)) mlp_tiles<true, double>(sm, x, t, y, o, ns);
  } else {
    mlp_tiles<false, df>(sm, x, t, y, nullptr, ns);
  }
}
static_assert(kSmA % 2 == 0, "the squares are stored as doubles");

// Gradient g = sum of the CTAs' parts, in CTA order (FP64), and loss = the sum
// of the squares / ns; with m != NULL the gradient goes straight into an Adam
// step (Kingma & Ba) of the weights instead: m = b1 m + (1-b1) g;
// v = b2 v + (1-b2) g^2; w -= lr * mhat / (sqrt(vhat) + 1e-8)
__global__ void k_mlp_reduce(const double* __restrict__ part, int ncta, int ns, float* __restrict__ g,
                             float* __restrict__ loss, float* __restrict__ w, float* __restrict__ m,
                             float* __restrict__ v, float lr, float c1, float c2) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e > IFMM_MLP_NWEIGHTS) return;
  double s = 0.0;
#pragma unroll 8
  for (int c = 0; c < ncta; ++c) s += part[(long)c * (IFMM_MLP_NWEIGHTS + 1) + e];
  if (e == IFMM_MLP_NWEIGHTS) {
    if (loss) *loss = (float)(s / (double)ns);
    return;
  }
  const float gr = (float)s;
  if (g) g[e] = gr;
  if (!m) return;
  const float b1 = 0.9f, b2 = 0.999f;
  m[e] = b1 * m[e] + (1.f - b1) * gr;
  v[e] = b2 * v[e] + (1.f - b2) * gr * gr;
  const float mh = m[e] / c1, vh = v[e] / c2;
  w[e] -= lr * mh / (sqrtf(vh) + 1e-8f);
}

// counter-based initialisation: SplitMix64 (Steele, Lea, Flood) of (seed, index)
// -> uniform in [-a, a]
__global__ void k_mlp_init(float* __restrict__ w, int n, unsigned long long seed, float a, int first, int count) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  unsigned long long z = seed + 0x9E3779B97F4A7C15ull * (unsigned long long)(first + i + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  z = z ^ (z >> 31);
  const float u = (float)((z >> 40) * (1.0 / 16777216.0));  // [0, 1)
  w[first + i] = a * (2.f * u - 1.f);
  (void)n;
}

// Device memory of one call, carved from a single allocation (each allocation
// and release costs about as much as the kernels of a small call).
struct MlpBuffers {
  char* base = nullptr;
  size_t off = 0;
  static size_t up(size_t b) { return (b + 255) & ~(size_t)255; }
  explicit MlpBuffers(size_t bytes) { CKM(device_malloc((void**)&base, std::max<size_t>(bytes, 256))); }
  MlpBuffers(const MlpBuffers&) = delete;
  MlpBuffers& operator=(const MlpBuffers&) = delete;
  ~MlpBuffers() { cudaFree(base); }
  template <class T = float>
  T* get(size_t n) {
    T* p = (T*)(base + off);
    off += up(sizeof(T) * n);
    return p;
  }
};

// CTAs of a pass over ns samples: every tile its own CTA up to one CTA per SM
// (the shared memory of a CTA leaves room for one); fixed by ns, so that the
// order of the sums is.
static int mlp_ctas(int ns) { return std::min(152, (ns + kT - 1) / kT); }

static void mlp_attrs() {
  static PerDevice<std::once_flag> once;
  std::call_once(once(), [] {
    CKM(cudaFuncSetAttribute(k_mlp<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mlp_smem_bytes(false)));
    CKM(cudaFuncSetAttribute(k_mlp<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mlp_smem_bytes(true)));
  });
}

static void mlp_forward(const float* w, const float* x, float* y, int ns, cudaStream_t s) {
  if (ns <= 0) return;
  mlp_attrs();
  // forward alone needs 88 KB: two CTAs per SM
  k_mlp<false><<<std::min(2 * 152, (ns + kT - 1) / kT), kMlpThreads, mlp_smem_bytes(false), s>>>(w, x, nullptr, y,
                                                                                                nullptr, ns);
  CKM(cudaGetLastError());
}

static size_t mlp_part_doubles(int ns) { return (size_t)mlp_ctas(ns) * (IFMM_MLP_NWEIGHTS + 1); }

// loss and gradient over ns samples (g, loss may be NULL), or an Adam step of w
static void mlp_gradient(float* w, const float* x, const float* t, int ns, double* part, float* g, float* loss,
                         float* m, float* v, float lr, float c1, float c2, cudaStream_t s) {
  mlp_attrs();
  const int nc = mlp_ctas(ns);
  k_mlp<true><<<nc, kMlpThreads, mlp_smem_bytes(true), s>>>(w, x, t, nullptr, part, ns);
  k_mlp_reduce<<<(IFMM_MLP_NWEIGHTS + 1 + 63) / 64, 64, 0, s>>>(part, nc, ns, g, loss, w, m, v, lr, c1, c2);
  CKM(cudaGetLastError());
}

void mlp_predict_device(const float* d_w, const float* d_x, float* d_y, int ns, cudaStream_t s) {
  mlp_forward(d_w, d_x, d_y, ns, s);
}

}  // namespace ifmm

using namespace ifmm;

extern "C" {

ifmm_status ifmm_mlp_forward(const float* weights, const float* x, int64_t n, float* y, void* stream) {
  try {
    IFMM_REQUIRE(weights && x && y && n >= 0 && n < (1 << 26), IFMM_EINVAL, "bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    MlpBuffers B(4 * (MlpBuffers::up(IFMM_MLP_NWEIGHTS) + MlpBuffers::up(n * kIn) + MlpBuffers::up(n)));
    float* dw = B.get(IFMM_MLP_NWEIGHTS);
    float* dx = B.get(n * kIn);
    float* dy = B.get(n);
    CKM(cudaMemcpyAsync(dw, weights, sizeof(float) * IFMM_MLP_NWEIGHTS, cudaMemcpyHostToDevice, s));
    CKM(cudaMemcpyAsync(dx, x, sizeof(float) * n * kIn, cudaMemcpyHostToDevice, s));
    mlp_forward(dw, dx, dy, (int)n, s);
    CKM(cudaMemcpyAsync(y, dy, sizeof(float) * n, cudaMemcpyDeviceToHost, s));
    CKM(cudaStreamSynchronize(s));
    return IFMM_OK;
  } catch (const Error& e) {
    set_last_error(e.what());
    return e.code;
  }
}

ifmm_status ifmm_mlp_grad(const float* weights, const float* x, const float* t, int64_t n, float* grad, float* loss,
                          void* stream) {
  try {
    IFMM_REQUIRE(weights && x && t && grad && n >= 1 && n < (1 << 26), IFMM_EINVAL, "bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    const size_t np = mlp_part_doubles((int)n);
    MlpBuffers B(4 * (MlpBuffers::up(IFMM_MLP_NWEIGHTS) + MlpBuffers::up(IFMM_MLP_NWEIGHTS + 1) +
                      MlpBuffers::up(n * kIn) + MlpBuffers::up(n)) +
                 MlpBuffers::up(8 * np));
    float* dw = B.get(IFMM_MLP_NWEIGHTS);
    float* dg = B.get(IFMM_MLP_NWEIGHTS + 1);  // the loss after the gradient
    float* dx = B.get(n * kIn);
    float* dt = B.get(n);
    double* part = B.get<double>(np);
    CKM(cudaMemcpyAsync(dw, weights, sizeof(float) * IFMM_MLP_NWEIGHTS, cudaMemcpyHostToDevice, s));
    CKM(cudaMemcpyAsync(dx, x, sizeof(float) * n * kIn, cudaMemcpyHostToDevice, s));
    CKM(cudaMemcpyAsync(dt, t, sizeof(float) * n, cudaMemcpyHostToDevice, s));
    mlp_gradient(dw, dx, dt, (int)n, part, dg, dg + IFMM_MLP_NWEIGHTS, nullptr, nullptr, 0.f, 1.f, 1.f, s);
    float hl = 0.f;
    CKM(cudaMemcpyAsync(grad, dg, sizeof(float) * IFMM_MLP_NWEIGHTS, cudaMemcpyDeviceToHost, s));
    CKM(cudaMemcpyAsync(&hl, dg + IFMM_MLP_NWEIGHTS, sizeof(float), cudaMemcpyDeviceToHost, s));
    CKM(cudaStreamSynchronize(s));
    if (loss) *loss = hl;
    return IFMM_OK;
  } catch (const Error& e) {
    set_last_error(e.what());
    return e.code;
  }
}

ifmm_status ifmm_mlp_train(const float* x, const float* t, int64_t n, int epochs, int batch, float lr, uint64_t seed,
                           float* weights, float* final_loss, void* stream) {
  try {
    IFMM_REQUIRE(x && t && weights && n >= 1 && n < (1 << 26) && epochs >= 1 && batch >= 1, IFMM_EINVAL,
                 "bad argument");
    cudaStream_t s = (cudaStream_t)stream;
    const int bs = (int)std::min<int64_t>(batch, n);
    const size_t np = mlp_part_doubles((int)n);  // the largest pass: the final loss, over every row
    MlpBuffers B(4 * (4 * MlpBuffers::up(IFMM_MLP_NWEIGHTS + 1) + MlpBuffers::up(n * kIn) + MlpBuffers::up(n)) +
                 MlpBuffers::up(8 * np));
    float* dw = B.get(IFMM_MLP_NWEIGHTS);
    float* dm = B.get(IFMM_MLP_NWEIGHTS);
    float* dv = B.get(IFMM_MLP_NWEIGHTS);
    float* dl = B.get(1);
    float* dx = B.get((size_t)n * kIn);
    float* dt = B.get(n);
    double* part = B.get<double>(np);
    CKM(cudaMemcpyAsync(dx, x, sizeof(float) * n * kIn, cudaMemcpyHostToDevice, s));
    CKM(cudaMemcpyAsync(dt, t, sizeof(float) * n, cudaMemcpyHostToDevice, s));
    CKM(cudaMemsetAsync(dm, 0, sizeof(float) * IFMM_MLP_NWEIGHTS, s));
    CKM(cudaMemsetAsync(dv, 0, sizeof(float) * IFMM_MLP_NWEIGHTS, s));
    // He-uniform weights, zero biases
    CKM(cudaMemsetAsync(dw, 0, sizeof(float) * IFMM_MLP_NWEIGHTS, s));
    for (int l = 0; l < 4; ++l) {
      int wo, bo;
      layer_offsets(l, &wo, &bo);
      const int cnt = kDims[l] * kDims[l + 1];
      const float a = std::sqrt(6.0f / (float)kDims[l]);
      k_mlp_init<<<(cnt + 255) / 256, 256, 0, s>>>(dw, IFMM_MLP_NWEIGHTS, (unsigned long long)seed, a, wo, cnt);
    }
    long step = 0;
    const int nb = (int)((n + bs - 1) / bs);
    for (int ep = 0; ep < epochs; ++ep)
      for (int bi = 0; bi < nb; ++bi) {
        const int64_t off = (int64_t)bi * bs;
        const int cur = (int)std::min<int64_t>(bs, n - off);
        ++step;
        const float c1 = 1.f - std::pow(0.9f, (float)step), c2 = 1.f - std::pow(0.999f, (float)step);
        mlp_gradient(dw, dx + off * kIn, dt + off, cur, part, nullptr, nullptr, dm, dv, lr, c1, c2, s);
      }
    CKM(cudaMemcpyAsync(weights, dw, sizeof(float) * IFMM_MLP_NWEIGHTS, cudaMemcpyDeviceToHost, s));
    CKM(cudaStreamSynchronize(s));
    if (final_loss) {
      // loss over the whole set with the final weights
      mlp_gradient(dw, dx, dt, (int)n, part, nullptr, dl, nullptr, nullptr, 0.f, 1.f, 1.f, s);
      CKM(cudaMemcpyAsync(final_loss, dl, sizeof(float), cudaMemcpyDeviceToHost, s));
      CKM(cudaStreamSynchronize(s));
    }
    return IFMM_OK;
  } catch (const Error& e) {
    set_last_error(e.what());
    return e.code;
  }
}

}  // extern "C"
