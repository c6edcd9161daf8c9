// A CUDA runtime without a GPU, preloaded before libcudart by the CPU tests of
// what the library asks of the runtime: allocations are host memory, copies
// are memcpy, kernels do not run.  Devices are numbered by fake_set_device.
// Each launch is recorded and is held to the runtime's rule on dynamic shared
// memory: no more than cudaFuncAttributeMaxDynamicSharedMemorySize as last set
// for that kernel on the current device, 48 KB where it was never set.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <utility>
#include <vector>

namespace {
struct Launch {
  int dev;
  std::string name;
  size_t smem;
  bool refused;
  int carveout;  // preferred share of shared memory in percent, -1 without one
};
std::mutex mu;
std::map<const void*, std::string>& names() {  // built before any static constructor registers a kernel
  static std::map<const void*, std::string> m;
  return m;
}
std::map<std::pair<const void*, int>, size_t> limit;
std::map<const char*, std::pair<size_t, int>> memory;  // device allocations: start -> (bytes, device)
std::vector<Launch> launches;
std::map<std::pair<const void*, int>, void*> symbols;
int device = 0;
const size_t kDefault = 48 * 1024, kOptin = 227 * 1024, kSm = 228 * 1024;
thread_local struct { dim3 grid, block; size_t smem; cudaStream_t s; } call;

cudaError_t launch(const void* f, size_t smem, int carveout = -1) {
  std::lock_guard<std::mutex> lk(mu);
  auto it = limit.find({f, device});
  const bool refused = smem > (it == limit.end() ? kDefault : it->second);
  auto n = names().find(f);
  launches.push_back({device, n == names().end() ? "?" : n->second, smem, refused, carveout});
  return refused ? cudaErrorInvalidValue : cudaSuccess;
}
cudaError_t allocate(void** p, size_t n) {
  std::lock_guard<std::mutex> lk(mu);
  *p = aligned_alloc(256, (n + 255) / 256 * 256 + 256);
  if (!*p) return cudaErrorMemoryAllocation;
  memset(*p, 0, n);
  memory[static_cast<char*>(*p)] = {n, device};
  return cudaSuccess;
}
int encode_tiled(...) { return 0; }
char token[64];  // handles of streams, events and graphs
}  // namespace

extern "C" {
// ---- the tests' own view
void fake_set_device(int d) { device = d; }
void* fake_alloc(size_t n) {
  void* p = nullptr;
  allocate(&p, n);
  return p;
}
int fake_launches(void) { return (int)launches.size(); }
int fake_carveout(int i) { return launches[i].carveout; }
const char* fake_launch(int i, int* dev, size_t* smem, int* refused) {
  *dev = launches[i].dev;
  *smem = launches[i].smem;
  *refused = launches[i].refused;
  return launches[i].name.c_str();
}

// ---- registration and launches
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(token); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
  call = {grid, block, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  *grid = call.grid;
  *block = call.block;
  *smem = call.smem;
  *static_cast<cudaStream_t*>(s) = call.s;
  return cudaSuccess;
}
static thread_local cudaError_t last = cudaSuccess;
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  const cudaError_t e = launch(reinterpret_cast<const void*>(k), smem);
  if (e != cudaSuccess) last = e;
  return e;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  int carveout = -1;
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributePreferredSharedMemoryCarveout) carveout = (int)c->attrs[i].val.sharedMemCarveout;
  const cudaError_t e = launch(f, c->dynamicSmemBytes, carveout);
  if (e != cudaSuccess) last = e;
  return e;
}
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::mutex> lk(mu);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (v < 0 || (size_t)v > kOptin) return cudaErrorInvalidValue;
    limit[{f, device}] = (size_t)v;
  }
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int threads, size_t smem,
                                                                   unsigned) {
  *n = (int)(kSm / (smem + 1024));
  if (*n > 2048 / threads) *n = 2048 / threads;
  return cudaSuccess;
}

// ---- devices, memory, streams, events, graphs
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }  // worker threads take the one device the test has set
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  switch (a) {
    case cudaDevAttrMultiProcessorCount: *v = 152; break;
    case cudaDevAttrL2CacheSize: *v = 129 << 20; break;
    case cudaDevAttrCooperativeLaunch: *v = 1; break;
    case cudaDevAttrMaxSharedMemoryPerBlockOptin: *v = (int)kOptin; break;
    default: *v = 0;
  }
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
  void*& a = symbols[{symbol, device}];
  if (!a) allocate(&a, 8 << 20);
  *p = a;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return allocate(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return allocate(p, n); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return (*p = calloc(1, n)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) {
  std::lock_guard<std::mutex> lk(mu);
  memory.erase(static_cast<char*>(p));
  free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* at, const void* p) {
  std::lock_guard<std::mutex> lk(mu);
  *at = cudaPointerAttributes{};
  auto it = memory.upper_bound(static_cast<const char*>(p));
  if (it != memory.begin()) {
    --it;
    if (static_cast<const char*>(p) < it->first + it->second.first) {
      at->type = cudaMemoryTypeDevice;
      at->device = it->second.second;
    }
  }
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = reinterpret_cast<cudaStream_t>(token); return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = reinterpret_cast<cudaGraph_t>(token); return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = reinterpret_cast<cudaEvent_t>(token); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1.f; return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { *e = reinterpret_cast<cudaGraphExec_t>(token); return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *f = reinterpret_cast<void*>(&encode_tiled);
  *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}  // extern "C"
