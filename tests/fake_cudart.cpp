// CUDA runtime without a GPU, for tests of the library's host code: two devices
// whose memory is host memory, copies that are done at once, kernels that do
// nothing.  It refuses what a device would refuse (a launch with more dynamic
// shared memory than its function was allowed on that device, an allocation
// beyond the device's memory) and records copies and launches, and work on
// another stream that does not wait for the null stream's.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>

#define API extern "C" __attribute__((visibility("default")))

namespace {
struct Block {
  size_t n;
  int device;
};
constexpr int kDevices = 2;
int g_device = 0;
cudaError_t g_last = cudaSuccess;
std::map<uintptr_t, Block> g_blocks;
size_t g_used[kDevices], g_total[kDevices] = {(size_t)1 << 38, (size_t)1 << 38};
std::map<std::pair<int, const void*>, int> g_smem;   // function's dynamic shared memory on a device
std::map<const void*, std::string> g_names;
std::string g_log;
bool g_capturing = false, g_null_pending = false;
int g_unordered = 0;
struct Call {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} g_call;

cudaError_t done(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}
const std::pair<const uintptr_t, Block>* find(const void* p) {
  auto it = g_blocks.upper_bound((uintptr_t)p);
  if (it == g_blocks.begin()) return nullptr;
  --it;
  return (uintptr_t)p < it->first + it->second.n ? &*it : nullptr;
}
// work on a stream: the null stream's own is pending until something waits for it
void work(cudaStream_t s) {
  if (g_capturing) return;
  if (!s)
    g_null_pending = true;
  else if (g_null_pending)
    ++g_unordered;
}
cudaError_t launch(const void* f, size_t smem, cudaStream_t s) {
  work(s);
  auto it = g_smem.find({g_device, f});
  if (smem > 48 * 1024 && (it == g_smem.end() || (size_t)it->second < smem)) return done(cudaErrorInvalidValue);
  g_log += "launch " + std::to_string(g_device) + " " + g_names[f] + "\n";
  return cudaSuccess;
}
cudaError_t copy(void* d, const void* s, size_t n, cudaStream_t st) {
  work(st);
  std::memmove(d, s, n);
  g_log += "copy " + std::to_string((uintptr_t)d) + " " + std::to_string((uintptr_t)s) + " " + std::to_string(n) + "\n";
  return cudaSuccess;
}
CUresult CUDAAPI encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                        const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                        CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
template <typename T>
cudaError_t handle(T* p) {   // something to hold and to destroy
  *p = reinterpret_cast<T>(std::malloc(1));
  return cudaSuccess;
}
}  // namespace

// for the tests
API void fake_set_total(int device, size_t bytes) { g_total[device] = bytes; }
API size_t fake_used(int device) { return g_used[device]; }
API int fake_unordered() { return g_unordered; }
API void fake_clear_log() { g_log.clear(); }
API const char* fake_log() { return g_log.c_str(); }

// devices, memory
API cudaError_t cudaGetDeviceCount(int* n) { return *n = kDevices, cudaSuccess; }
API cudaError_t cudaSetDevice(int d) {
  if (d < 0 || d >= kDevices) return done(cudaErrorInvalidDevice);
  g_device = d;
  return cudaSuccess;
}
API cudaError_t cudaGetDevice(int* d) { return *d = g_device, cudaSuccess; }
API cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int device) {
  *v = a == cudaDevAttrComputeCapabilityMajor ? 10 : a == cudaDevAttrComputeCapabilityMinor ? 3 : device ? 76 : 152;
  return cudaSuccess;
}
API cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  p->major = 10;
  p->minor = 3;
  p->multiProcessorCount = 152;
  p->sharedMemPerBlockOptin = 227 * 1024;
  return cudaSuccess;
}
API cudaError_t cudaMemGetInfo(size_t* avail, size_t* total) {
  *total = g_total[g_device];
  *avail = *total - (g_used[g_device] < *total ? g_used[g_device] : *total);
  return cudaSuccess;
}
API cudaError_t cudaMalloc(void** p, size_t n) {
  *p = nullptr;
  if (g_used[g_device] + n > g_total[g_device]) return done(cudaErrorMemoryAllocation);
  *p = std::aligned_alloc(256, (n + 255) / 256 * 256);
  g_blocks[(uintptr_t)*p] = {n, g_device};
  g_used[g_device] += n;
  return cudaSuccess;
}
API cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  auto it = g_blocks.find((uintptr_t)p);
  if (it == g_blocks.end()) return done(cudaErrorInvalidValue);
  g_used[it->second.device] -= it->second.n;
  g_blocks.erase(it);
  std::free(p);
  return cudaSuccess;
}
API cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return *p = std::malloc(n), cudaSuccess; }
API cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
API cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::memset(a, 0, sizeof(*a));
  const auto* b = find(p);
  a->type = b ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  a->device = b ? b->second.device : -2;
  return cudaSuccess;
}
API cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) {
  copy(d, s, n, nullptr);
  g_null_pending = k != cudaMemcpyDeviceToHost;   // a copy from pageable memory may return before it has arrived
  return cudaSuccess;
}
API cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) { return copy(d, s, n, st); }
API cudaError_t cudaMemcpy2D(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind) {
  for (size_t i = 0; i < h; ++i) copy((char*)d + i * dp, (const char*)s + i * sp, w, nullptr);
  return cudaSuccess;
}
API cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t s) {
  work(s);
  if (!g_capturing) std::memset(p, v, n);
  return cudaSuccess;
}
API cudaError_t cudaMemset(void* p, int v, size_t n) { return cudaMemsetAsync(p, v, n, nullptr); }
API cudaError_t cudaGetSymbolAddress(void** p, const void* s) { return *p = const_cast<void*>(s), cudaSuccess; }

// errors, streams, events, graphs
API cudaError_t cudaGetLastError() { return std::exchange(g_last, cudaSuccess); }
API const char* cudaGetErrorName(cudaError_t) { return "error"; }
API cudaError_t cudaDeviceSynchronize() { return g_null_pending = false, cudaSuccess; }
API cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  if (!s) g_null_pending = false;
  return cudaSuccess;
}
API cudaError_t cudaDeviceGetStreamPriorityRange(int* lo, int* hi) { return *lo = 0, *hi = -1, cudaSuccess; }
API cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
API cudaError_t cudaStreamCreateWithPriority(cudaStream_t* s, unsigned, int) { return handle(s); }
API cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
API cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
API cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
API cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
API cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
API cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
API cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
API cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
API cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return g_capturing = true, cudaSuccess; }
API cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return g_capturing = false, handle(g); }
API cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) { return handle(e); }
API cudaError_t cudaGraphDestroy(cudaGraph_t g) { return std::free(g), cudaSuccess; }
API cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return std::free(e), cudaSuccess; }
API cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) {
  work(s);
  g_log += "graph\n";
  return cudaSuccess;
}
API cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                                 cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

// kernels
API cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_device, f}] = v;
  return cudaSuccess;
}
API cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  return *n = 152 / (int)c->gridDim.x, cudaSuccess;
}
API cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->dynamicSmemBytes, c->stream);
}
API cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  return *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f)), cudaSuccess;
}
API cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t s) {
  return launch(reinterpret_cast<const void*>(k), smem, s);
}
API unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
  g_call = {grid, block, smem, s};
  return 0;
}
API cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  *grid = g_call.grid;
  *block = g_call.block;
  *smem = g_call.smem;
  *static_cast<cudaStream_t*>(s) = g_call.stream;
  return cudaSuccess;
}
API void** __cudaRegisterFatBinary(void*) {
  static void* h = nullptr;
  return &h;
}
API void __cudaRegisterFatBinaryEnd(void**) {}
API void __cudaUnregisterFatBinary(void**) {}
API void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
API void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_names[f] = name;
}
