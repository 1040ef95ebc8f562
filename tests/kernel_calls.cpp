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
}
