// A CUDA runtime on the host for tests of the library's host code: device
// memory is host memory (zeroed), kernels do nothing, and chosen calls fail.
// Linked with the library's object files in place of the CUDA runtime. Launch
// and attribute calls follow the rules that the host code depends on: more
// than 48 KB of dynamic shared memory has to be allowed for the kernel on the
// current device.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <utility>

namespace {
int g_dev = 0, g_fail_alloc = 0, g_live = 0, g_ran = 0;
size_t g_limit = size_t(1) << 30;
cudaError_t g_last = cudaSuccess;
std::string g_fail_launch;
std::map<const void*, std::string> g_names;
std::map<std::pair<int, const void*>, int> g_smem;
std::set<void*> g_blocks;
struct { dim3 g, b; size_t smem; cudaStream_t s; } g_cfg;

cudaError_t keep(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}
cudaError_t alloc(void** p, size_t n) {
  *p = nullptr;
  if ((g_fail_alloc > 0 && --g_fail_alloc == 0) || n > g_limit) return keep(cudaErrorMemoryAllocation);
  *p = std::calloc(n ? n : 1, 1);
  g_blocks.insert(*p);
  ++g_live;
  return cudaSuccess;
}
cudaError_t launch(const void* f, dim3 grid, size_t smem) {
  const std::string& name = g_names[f];
  if (!g_fail_launch.empty() && name.find(g_fail_launch) != std::string::npos) return keep(cudaErrorLaunchFailure);
  if (grid.x == 0 || grid.y == 0 || grid.z == 0) return keep(cudaErrorInvalidConfiguration);
  const auto it = g_smem.find({g_dev, f});
  if (smem > 48 * 1024 && (it == g_smem.end() || smem > (size_t)it->second)) return keep(cudaErrorInvalidValue);
  ++g_ran;
  return cudaSuccess;
}
}  // namespace

extern "C" {
void fake_reset() {
  g_dev = g_fail_alloc = 0;
  g_last = cudaSuccess;
  g_fail_launch.clear();
}
void fake_device(int d) { g_dev = d; }
void fake_fail_alloc(int k) { g_fail_alloc = k; }          // the k-th allocation from now fails
void fake_fail_launch(const char* s) { g_fail_launch = s; }  // launches of kernels with s in their name fail
int fake_live() { return g_live; }
int fake_ran() { return g_ran; }

cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t* p, int) { *p = nullptr; return cudaSuccess; }
cudaError_t cudaMemPoolCreate(cudaMemPool_t* p, const cudaMemPoolProps*) {
  *p = reinterpret_cast<cudaMemPool_t>(&g_dev);
  return cudaSuccess;
}
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
cudaError_t cudaMemPoolTrimTo(cudaMemPool_t, size_t) { return cudaSuccess; }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return alloc(p, n); }
cudaError_t cudaMallocFromPoolAsync(void** p, size_t n, cudaMemPool_t, cudaStream_t) { return alloc(p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  if (g_blocks.erase(p) != 1) std::abort();   // not allocated, or freed twice
  std::free(p);
  --g_live;
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { *p = std::calloc(n, 1); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { std::free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { std::memset(d, v, n); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { *s = nullptr; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { *g = nullptr; return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = reinterpret_cast<cudaEvent_t>(&g_dev); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { *t = 0.f; return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { *p = nullptr; return cudaErrorNotSupported; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_smem[{g_dev, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { *n = 1; return cudaSuccess; }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3 g, dim3, void**, size_t smem, cudaStream_t) {
  return launch(f, g, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim, c->dynamicSmemBytes);
}

// what the compiler's launch and registration code calls
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, void*, void*, void*, void*, int*) {
  g_names[f] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  g_cfg = {g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = g_cfg.g;
  *b = g_cfg.b;
  *smem = g_cfg.smem;
  *static_cast<cudaStream_t*>(s) = g_cfg.s;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void**, size_t smem, cudaStream_t) {
  return launch(reinterpret_cast<const void*>(k), g, smem);
}
}
