// A stand-in for the CUDA runtime on a machine without a GPU: preloaded before
// libifmm.so, it gives the library's host code devices to talk to.  Device memory is
// host memory under a limit, kernels do nothing, and every launch is checked as
// the runtime would check it: more than 48 KB of dynamic shared memory, or a
// cluster of more than eight CTAs, needs the function's attribute on the device that
// is current.  The functions at the end set the devices up and report what ran.
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <set>
#include <string>
#include <utility>
#include <vector>

namespace {

struct Pool {
  int dev;
  size_t reserved = 0, used = 0;
};
struct Block {
  size_t size;
  int dev;
  Pool* pool;
};
struct Device {
  size_t limit = (size_t)1 << 40, malloced = 0;
  std::vector<Pool*> pools;
  int max_cluster = 16;
  size_t in_use() const {
    size_t s = malloced;
    for (auto* p : pools) s += p->reserved;
    return s;
  }
};
struct State {
  std::recursive_mutex mu;
  std::map<int, Device> dev;
  std::map<const char*, Block> blocks;
  std::map<const void*, std::string> names;
  std::map<const void*, void*> vars;
  std::map<const void*, size_t> var_size;
  std::map<std::pair<int, const void*>, int> smem;
  std::set<std::pair<int, const void*>> wide;
  std::vector<std::string> log;
  std::string bad;
  int ndev = 2;
};
State& S() {
  static State* s = new State();
  return *s;
}
thread_local int t_dev = 0;
thread_local cudaError_t t_err = cudaSuccess;
thread_local struct {
  dim3 g, b;
  size_t sm;
  void* st;
} t_cfg;
using Lock = std::lock_guard<std::recursive_mutex>;

cudaError_t fail(cudaError_t e) {
  t_err = e;
  return e;
}
cudaError_t launch(const void* f, unsigned grid, unsigned threads, size_t sm, unsigned cluster, bool run) {
  Lock l(S().mu);
  const std::string name = S().names.count(f) ? S().names[f] : "?";
  const auto a = S().smem.find({t_dev, f});
  const size_t lim = a == S().smem.end() ? 48 * 1024 : (size_t)a->second;
  const bool wide = cluster > 8;
  std::string why;
  if (!grid || !threads || threads > 1024) why = "grid or block";
  if (sm > lim) why = "dynamic shared memory";
  if (wide && !S().wide.count({t_dev, f})) why = "cluster size";
  if (cluster > (unsigned)S().dev[t_dev].max_cluster) why = run ? "cluster not resident" : "";
  if (!why.empty()) {
    S().bad += name + " on device " + std::to_string(t_dev) + ": " + why + "\n";
    return fail(cudaErrorInvalidValue);
  }
  if (run) S().log.push_back(name);
  return cudaSuccess;
}
cudaError_t take(void** p, size_t n, Pool* pool) {
  Lock l(S().mu);
  Device& D = S().dev[pool ? pool->dev : t_dev];
  const size_t more = pool ? (pool->used + n > pool->reserved ? pool->used + n - pool->reserved : 0) : n;
  if (D.in_use() + more > D.limit) return fail(cudaErrorMemoryAllocation);
  void* q = calloc(1, n + 256);
  if (!q) return fail(cudaErrorMemoryAllocation);
  if (pool) {
    pool->used += n;
    pool->reserved += more;
  } else {
    D.malloced += n;
  }
  *p = q;
  S().blocks[(const char*)q] = Block{n, pool ? pool->dev : t_dev, pool};
  return cudaSuccess;
}
cudaError_t give(void* p) {
  if (!p) return cudaSuccess;
  Lock l(S().mu);
  auto it = S().blocks.find((const char*)p);
  if (it == S().blocks.end()) return fail(cudaErrorInvalidValue);
  if (it->second.pool)
    it->second.pool->used -= it->second.size;
  else
    S().dev[it->second.dev].malloced -= it->second.size;
  S().blocks.erase(it);
  free(p);
  return cudaSuccess;
}

}  // namespace

extern "C" {

// ---------------------------------------------------------------- the runtime's entries
void** __cudaRegisterFatBinary(void*) {
  static void* h = nullptr;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  S().names[host] = name;
}
void __cudaRegisterVar(void**, char* host, char*, const char*, int, size_t size, int, int) { S().var_size[host] = size; }
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t sm, cudaStream_t st) {
  t_cfg = {g, b, sm, st};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* sm, void* st) {
  *g = t_cfg.g;
  *b = t_cfg.b;
  *sm = t_cfg.sm;
  *(void**)st = t_cfg.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t sm, cudaStream_t) {
  return launch((const void*)k, g.x * g.y * g.z, b.x * b.y * b.z, sm, 1, true);
}
static unsigned cluster_of(const cudaLaunchConfig_t* c) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension) return c->attrs[i].val.clusterDim.x;
  return 1;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim.x * c->gridDim.y * c->gridDim.z, c->blockDim.x * c->blockDim.y * c->blockDim.z,
                c->dynamicSmemBytes, cluster_of(c), true);
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void* f, const cudaLaunchConfig_t* c) {
  *n = 0;
  const cudaError_t e = launch(f, 1, c->blockDim.x, c->dynamicSmemBytes, cluster_of(c), false);
  if (e == cudaSuccess) *n = cluster_of(c) <= (unsigned)S().dev[t_dev].max_cluster ? 4 : 0;
  return e;
}
cudaError_t cudaFuncSetAttribute(const void* f, enum cudaFuncAttribute a, int v) {
  Lock l(S().mu);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) S().smem[{t_dev, f}] = v;
  if (a == cudaFuncAttributeNonPortableClusterSizeAllowed && v) S().wide.insert({t_dev, f});
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(struct cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* v) {
  Lock l(S().mu);
  void*& q = S().vars[v];
  if (!q) q = calloc(1, 64);
  *p = q;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceCount(int* n) {
  *n = S().ndev;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = t_dev;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d >= S().ndev) return fail(cudaErrorInvalidDevice);
  t_dev = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, enum cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize(void) { return cudaSuccess; }
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = t_err;
  t_err = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }

cudaError_t cudaMalloc(void** p, size_t n) { return take(p, n, nullptr); }
cudaError_t cudaFree(void* p) { return give(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return give(p); }
cudaError_t cudaMallocHost(void** p, size_t n) {
  *p = calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const struct cudaMemPoolProps* pr) {
  Lock l(S().mu);
  Pool* q = new Pool{pr->location.id};
  S().dev[q->dev].pools.push_back(q);
  *p = (cudaMemPool_t)q;
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, enum cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolGetAttribute(cudaMemPool_t p, enum cudaMemPoolAttr a, void* v) {
  *(unsigned long long*)v = a == cudaMemPoolAttrReservedMemCurrent ? ((Pool*)p)->reserved : ((Pool*)p)->used;
  return cudaSuccess;
}
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t p, size_t keep) {
  Lock l(S().mu);
  Pool* q = (Pool*)p;
  if (q->reserved > keep) q->reserved = keep > q->used ? keep : q->used;
  return cudaSuccess;
}
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t pool, cudaStream_t) {
  return take(p, n, (Pool*)pool);
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, enum cudaMemcpyKind) {
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, enum cudaMemcpyKind, cudaStream_t) {
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(struct cudaPointerAttributes* a, const void* p) {
  Lock l(S().mu);
  memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeUnregistered;
  auto it = S().blocks.upper_bound((const char*)p);
  if (it != S().blocks.begin() && (const char*)p < (--it)->first + it->second.size) {
    a->type = cudaMemoryTypeDevice;
    a->device = it->second.dev;
  }
  return cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  free((void*)s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, enum cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = (cudaGraph_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = (cudaGraphExec_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
  free((void*)e);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  free((void*)g);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  free((void*)e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}

// ---------------------------------------------------------------- the tests' entries
void fake_set_device(int d) { t_dev = d; }
void fake_max_cluster(int d, int n) { S().dev[d].max_cluster = n; }
void fake_limit(int d, size_t bytes) { S().dev[d].limit = bytes; }
size_t fake_in_use(int d) { return S().dev[d].in_use(); }
void fake_clear(void) {
  S().log.clear();
  S().bad.clear();
}
// launches since fake_clear whose (mangled) kernel name contains s
int fake_launches(const char* s) {
  int n = 0;
  for (auto& x : S().log) n += x.find(s) != std::string::npos;
  return n;
}
// the refused launches since fake_clear
const char* fake_refused(void) { return S().bad.c_str(); }
}
