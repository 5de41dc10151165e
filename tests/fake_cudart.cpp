// A CUDA runtime on host memory, preloaded by test_host_paths.py in front of the real
// one: device memory is the process's, copies are memcpy, kernels do not run.  It
// counts what the tests ask about (launches, copies per buffer, work left unordered
// on the legacy stream), fails a chosen allocation and plants what the device would
// have copied back.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#define FAKE extern "C" __attribute__((visibility("default")))

namespace {
std::map<const char*, size_t> g_mem;  // device allocations
std::vector<const void*> g_foreign;   // buffers of another GPU
std::map<size_t, std::string> g_plant;
std::map<const void*, int> g_copies;
int g_legacy = 0, g_launches = 0, g_fail_at = 0, g_allocs = 0, g_memsets = 0;

bool on_device(const void* p) {
  auto it = g_mem.upper_bound(static_cast<const char*>(p));
  if (it == g_mem.begin()) return false;
  --it;
  return static_cast<const char*>(p) < it->first + it->second;
}
bool foreign(const void* p) {
  for (const void* q : g_foreign)
    if (q == p) return true;
  return false;
}
cudaError_t alloc(void** p, size_t n) {
  if (++g_allocs == g_fail_at) return cudaErrorMemoryAllocation;
  *p = calloc(1, n ? n : 1);
  g_mem[static_cast<char*>(*p)] = n ? n : 1;
  g_copies.erase(g_copies.lower_bound(*p), g_copies.lower_bound(static_cast<char*>(*p) + n));
  return cudaSuccess;
}
cudaError_t release(void* p) {
  if (p) g_mem.erase(static_cast<char*>(p));
  free(p);
  return cudaSuccess;
}
void copy(void* dst, const void* src, size_t n) {
  ++g_copies[dst];
  ++g_copies[src];
  auto it = g_plant.find(n);
  if (it != g_plant.end() && on_device(src) && !on_device(dst))
    memcpy(dst, it->second.data(), n);
  else
    memmove(dst, src, n);
}
cudaError_t launch() {
  ++g_launches;
  return cudaSuccess;
}
}  // namespace

// ------------------------------------------------------------- for the tests
FAKE int fake_legacy_pending() { return g_legacy; }
FAKE int fake_launches() { return g_launches; }
FAKE int fake_memsets_on_streams() { return g_memsets; }
FAKE void fake_fail_alloc(int nth) { g_allocs = 0, g_fail_at = nth; }
FAKE int fake_allocs() { return g_allocs; }
FAKE void fake_plant(size_t n, const void* data) {
  if (data)
    g_plant[n] = std::string(static_cast<const char*>(data), n);
  else
    g_plant.erase(n);
}
FAKE void fake_foreign(const void* p) { g_foreign.push_back(p); }
FAKE int fake_copies(const void* p) { return g_copies[p]; }

// ------------------------------------------------------------- memory
FAKE cudaError_t cudaMalloc(void** p, size_t n) { return alloc(p, n); }
FAKE cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return alloc(p, n); }
FAKE cudaError_t cudaFree(void* p) { return release(p); }
FAKE cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return release(p); }
FAKE cudaError_t cudaMallocHost(void** p, size_t n) { return *p = calloc(1, n), cudaSuccess; }
FAKE cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }
FAKE cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  copy(d, s, n);
  if (!st) ++g_legacy;
  return cudaSuccess;
}
// A copy to the host ends when the legacy stream has come to it; one to the device
// may return once its source has been staged.
FAKE cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  copy(d, s, n);
  g_legacy = on_device(d) ? g_legacy + 1 : 0;
  return cudaSuccess;
}
FAKE cudaError_t cudaMemset(void* p, int v, size_t n) { return memset(p, v, n), ++g_legacy, cudaSuccess; }
FAKE cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t st) {
  memset(p, v, n);
  ++(st ? g_memsets : g_legacy);
  return cudaSuccess;
}
FAKE cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof(*a));
  a->type = on_device(p) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  a->device = foreign(p) ? 1 : 0;
  a->devicePointer = const_cast<void*>(p);
  return cudaSuccess;
}
FAKE cudaError_t cudaGetSymbolAddress(void** p, const void*) { return alloc(p, 1 << 23); }

// ------------------------------------------------------------- device, streams, events
FAKE cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
FAKE cudaError_t cudaSetDevice(int) { return cudaSuccess; }
FAKE cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
FAKE cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) { return *p = nullptr, cudaSuccess; }
FAKE cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
FAKE cudaError_t cudaDeviceSynchronize() { return g_legacy = 0, cudaSuccess; }
FAKE cudaError_t cudaGetLastError() { return cudaSuccess; }
FAKE const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
FAKE cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  return *s = reinterpret_cast<cudaStream_t>(0x100), cudaSuccess;
}
FAKE cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
FAKE cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (!s) g_legacy = 0;
  return cudaSuccess;
}
FAKE cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
FAKE cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = reinterpret_cast<cudaEvent_t>(0x200), cudaSuccess; }
FAKE cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
FAKE cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
FAKE cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
FAKE cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
FAKE cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }

// ------------------------------------------------------------- graphs
FAKE cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
FAKE cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  return *g = reinterpret_cast<cudaGraph_t>(0x300), cudaSuccess;
}
FAKE cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  return *e = reinterpret_cast<cudaGraphExec_t>(0x400), cudaSuccess;
}
FAKE cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
FAKE cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
FAKE cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
FAKE cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t* n) { return *n = 0, cudaSuccess; }
FAKE cudaError_t cudaGraphNodeGetType(cudaGraphNode_t, cudaGraphNodeType* t) {
  return *t = cudaGraphNodeTypeKernel, cudaSuccess;
}

// ------------------------------------------------------------- kernels
FAKE cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
FAKE cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof(*a));
  a->numRegs = 64;
  return cudaSuccess;
}
FAKE cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 1, cudaSuccess;
}
FAKE cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return launch(); }
FAKE cudaError_t __cudaGetKernel(cudaKernel_t* k, const void*) {
  return *k = reinterpret_cast<cudaKernel_t>(0x500), cudaSuccess;
}
FAKE cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return launch(); }
FAKE unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
FAKE cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = *b = dim3(1, 1, 1);
  *s = 0;
  *static_cast<void**>(st) = nullptr;
  return cudaSuccess;
}
FAKE void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
FAKE void __cudaRegisterFatBinaryEnd(void**) {}
FAKE void __cudaUnregisterFatBinary(void**) {}
FAKE void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
FAKE void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
