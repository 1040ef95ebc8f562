// The library's internal launchers on host arrays, for tests of what no public entry
// reaches by itself: built into a shared object next to libifmm.so by
// tests/kernel_calls.py.  Every function returns 0, or the library's status.
#include <cstring>
#include <vector>

#include "ifmm_kernels.h"
#include "runtime.h"

using namespace ifmm;

namespace {
template <class F>
int guarded(F&& f) {
  try {
    f();
    return 0;
  } catch (const Error& e) {
    set_last_error(e.what());
    return e.code;
  }
}
}  // namespace

extern "C" {

// nmat matrices of orders n[i] back to back, each replaced by its inverse
int kc_inv(int nmat, const int* n, double* A, int* info) {
  return guarded([&] {
    DescStage st;
    cudaStream_t s;
    CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    st.stream = s;
    size_t tot = 0;
    for (int i = 0; i < nmat; ++i) tot += (size_t)n[i] * n[i];
    DeviceArena mem;
    double* dA = mem.alloc(tot + 1);
    int* di = (int*)mem.alloc_bytes(sizeof(int) * nmat);
    CK(cudaMemcpyAsync(dA, A, sizeof(double) * tot, cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(di, info, sizeof(int) * nmat, cudaMemcpyHostToDevice, s));
    std::vector<InvDesc> v;
    size_t off = 0;
    for (int i = 0; i < nmat; ++i) {
      v.push_back(InvDesc{dA + off, n[i] > 0 ? n[i] : 1, n[i], di + i, 0});
      off += (size_t)n[i] * n[i];
    }
    launch_inv(st, v);
    CK(cudaMemcpyAsync(A, dA, sizeof(double) * tot, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(info, di, sizeof(int) * nmat, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    CK(cudaStreamDestroy(s));
  });
}

// one-sided Jacobi of the n x n matrix A (column-major), explicit (no pivoted R): the
// sorted singular values and the normalised columns
int kc_svd(int fp32, int n, const double* A, double* V, double* sig) {
  return guarded([&] {
    DescStage st;
    cudaStream_t s;
    CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    st.stream = s;
    DeviceArena mem;
    const size_t nn = (size_t)n * n;
    double *dA = mem.alloc(nn), *dV = mem.alloc(nn), *dw = mem.alloc(nn), *ds = mem.alloc(n);
    int* dk = (int*)mem.alloc_bytes(sizeof(int));
    CK(cudaMemcpyAsync(dA, A, sizeof(double) * nn, cudaMemcpyHostToDevice, s));
    CK(cudaMemcpyAsync(dk, &n, sizeof(int), cudaMemcpyHostToDevice, s));
    SvdRtDesc d{};
    d.A = dA;
    d.ld = n;
    d.n = n;
    d.kin = dk;
    d.jpvt = nullptr;
    d.V = dV;
    d.ldv = n;
    d.sig = ds;
    d.work = dw;
    launch_svd_rt(st, std::vector<SvdRtDesc>{d}, fp32 ? P32 : P64);
    CK(cudaMemcpyAsync(V, dV, sizeof(double) * nn, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(sig, ds, sizeof(double) * n, cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    CK(cudaStreamDestroy(s));
  });
}

// X = the inverse of the n x n matrix A (column-major) as the level-1 system's is
// formed; columns: by the launches per column
int kc_top_inverse(int n, const double* A, double* X, int* info, int columns) {
  return guarded([&] {
    cudaStream_t s;
    CK(cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking));
    DeviceArena mem;
    const size_t nn = (size_t)n * n;
    double *dA = mem.alloc(nn), *dX = mem.alloc(nn), *dw = mem.alloc(big_inverse_work_doubles(n));
    int *dp = (int*)mem.alloc_bytes(sizeof(int) * n), *di = (int*)mem.alloc_bytes(sizeof(int));
    CK(cudaMemcpyAsync(dA, A, sizeof(double) * nn, cudaMemcpyHostToDevice, s));
    big_inverse(s, dA, n, dX, dp, dw, di, columns != 0);
    CK(cudaMemcpyAsync(X, dX, sizeof(double) * nn, cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(info, di, sizeof(int), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    CK(cudaStreamDestroy(s));
  });
}
}
