// Device and pinned-host memory kept between calls (declared in runtime.h).
#include <cuda_runtime.h>

#include <exception>
#include <map>
#include <mutex>
#include <unordered_map>

#include "runtime.h"

namespace ifmm {

namespace {

constexpr size_t kDeviceKeep = (size_t)16 << 30;
constexpr size_t kPinnedKeep = (size_t)256 << 20;

struct DevicePool {
  cudaMemPool_t pool = nullptr;
  cudaStream_t stream = nullptr;  // allocations and releases only: never any work
};

struct State {
  std::mutex mu;
  std::map<int, DevicePool> dev;
  std::unordered_map<void*, int> owner;      // device block -> device
  std::multimap<size_t, void*> pinned;       // unused pinned chunks by size
  size_t pinned_bytes = 0;
  long trees = 0;
};
State& state() {
  static State* s = new State();  // never destroyed: handles may be freed during the process' end
  return *s;
}

DevicePool& device_pool(State& S, int dev) {
  DevicePool& P = S.dev[dev];
  if (!P.pool) {
    cudaMemPoolProps pr = {};
    pr.allocType = cudaMemAllocationTypePinned;
    pr.location.type = cudaMemLocationTypeDevice;
    pr.location.id = dev;
    CK(cudaMemPoolCreate(&P.pool, &pr));
    // what stays is bounded by pool_free, not by the driver at every
    // synchronization (which unmaps and remaps blocks in the middle of a job)
    unsigned long long keep = ~0ull;
    CK(cudaMemPoolSetAttribute(P.pool, cudaMemPoolAttrReleaseThreshold, &keep));
    CK(cudaStreamCreateWithFlags(&P.stream, cudaStreamNonBlocking));
  }
  return P;
}

void drop_pinned(State& S) {
  for (auto& c : S.pinned) cudaFreeHost(c.second);
  S.pinned.clear();
  S.pinned_bytes = 0;
}

// gives the device memory kept unused on dev back to the driver
void trim(State& S, int dev) {
  auto it = S.dev.find(dev);
  if (it == S.dev.end() || !it->second.pool) return;
  cudaStreamSynchronize(it->second.stream);
  cudaMemPoolTrimTo(it->second.pool, 0);
}

}  // namespace

cudaError_t device_malloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e != cudaErrorMemoryAllocation) return e;
  cudaGetLastError();
  State& S = state();
  std::lock_guard<std::mutex> lock(S.mu);
  int dev = 0;
  if (cudaGetDevice(&dev) == cudaSuccess) trim(S, dev);
  e = cudaMalloc(p, bytes);
  if (e != cudaSuccess) cudaGetLastError();
  return e;
}

void* pool_alloc(size_t bytes) {
  State& S = state();
  std::lock_guard<std::mutex> lock(S.mu);
  int dev = 0;
  CK(cudaGetDevice(&dev));
  DevicePool& P = device_pool(S, dev);
  void* p = nullptr;
  cudaError_t e = cudaMallocFromPoolAsync(&p, bytes, P.pool, P.stream);
  if (e == cudaErrorMemoryAllocation) {  // give back what is kept and try once more
    cudaGetLastError();
    trim(S, dev);
    e = cudaMallocFromPoolAsync(&p, bytes, P.pool, P.stream);
  }
  if (e != cudaSuccess) cudaGetLastError();
  CK(e);
  CK(cudaStreamSynchronize(P.stream));  // usable on every stream from here on
  S.owner[p] = dev;
  return p;
}

void pool_free(void* p) {
  if (!p) return;
  State& S = state();
  std::lock_guard<std::mutex> lock(S.mu);
  auto it = S.owner.find(p);
  if (it == S.owner.end()) return;
  DevicePool& P = S.dev[it->second];
  S.owner.erase(it);
  cudaFreeAsync(p, P.stream);
  unsigned long long held = 0, used = 0;
  if (cudaMemPoolGetAttribute(P.pool, cudaMemPoolAttrReservedMemCurrent, &held) == cudaSuccess &&
      cudaMemPoolGetAttribute(P.pool, cudaMemPoolAttrUsedMemCurrent, &used) == cudaSuccess &&
      held > used + kDeviceKeep) {
    cudaStreamSynchronize(P.stream);
    cudaMemPoolTrimTo(P.pool, used + kDeviceKeep);
  }
}

void* pinned_alloc(size_t bytes, size_t* got) {
  State& S = state();
  {
    std::lock_guard<std::mutex> lock(S.mu);
    auto it = S.pinned.lower_bound(bytes);
    if (it != S.pinned.end() && it->first <= 16 * bytes) {
      void* p = it->second;
      *got = it->first;
      S.pinned_bytes -= it->first;
      S.pinned.erase(it);
      return p;
    }
  }
  void* p = nullptr;
  cudaError_t e = cudaMallocHost(&p, bytes);
  if (e == cudaErrorMemoryAllocation) {  // give back what is kept and try once more
    cudaGetLastError();
    {
      std::lock_guard<std::mutex> lock(S.mu);
      drop_pinned(S);
    }
    e = cudaMallocHost(&p, bytes);
  }
  if (e != cudaSuccess) cudaGetLastError();
  CK(e);
  *got = bytes;
  return p;
}

void pinned_free(void* p, size_t got) {
  if (!p) return;
  State& S = state();
  {
    std::lock_guard<std::mutex> lock(S.mu);
    if (S.trees > 0 && S.pinned_bytes + got <= kPinnedKeep) {
      S.pinned.emplace(got, p);
      S.pinned_bytes += got;
      return;
    }
  }
  cudaFreeHost(p);
}

void pool_tree_count(int delta) {
  State& S = state();
  std::lock_guard<std::mutex> lock(S.mu);
  S.trees += delta;
  if (S.trees > 0) return;
  drop_pinned(S);
  for (auto& d : S.dev) trim(S, d.first);
}

void pool_quiesce() {
  if (std::uncaught_exceptions() > 0) cudaDeviceSynchronize();
}

}  // namespace ifmm
