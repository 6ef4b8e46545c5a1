// A CUDA runtime on the host for the library's object files: memory is host
// memory, a launch only records its kernel, and every device keeps its own
// kernel attributes, as real devices do.  So the calls' routes (which kernels a
// solve launches) and their behaviour on a second device or after a refused
// attribute can be tested without a GPU.  Nothing a kernel would write is
// written; page-locked memory starts as 1.0, which a residual check reads as
// ||r|| = ||b||.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <utility>
#include <vector>

namespace {
int g_dev = 0;
cudaError_t g_last = cudaSuccess;
std::string g_refuse, g_fail;
std::map<const void*, std::string> g_names;
std::map<std::pair<int, const void*>, size_t> g_smem;   // opt-in per (device, kernel)
std::vector<std::string> g_launches;

cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}
cudaError_t launch(const void* f, size_t smem) {
  if (!g_fail.empty() && g_names[f].find(g_fail) != std::string::npos) return set(cudaErrorLaunchOutOfResources);
  if (smem > 48 * 1024) {
    const auto it = g_smem.find({g_dev, f});
    if (it == g_smem.end() || it->second < smem) return set(cudaErrorInvalidValue);
  }
  g_launches.push_back(g_names[f]);
  return cudaSuccess;
}
int encode_tiled(...) { return 0; }
template <class T>
cudaError_t handle(T* out) {
  *out = reinterpret_cast<T>(malloc(1));
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- the test's side
void fake_device(int dev) { g_dev = dev; }
void fake_refuse(const char* part) { g_refuse = part; }   // kernels whose opt-in fails
void fake_fail(const char* part) { g_fail = part; }       // kernels whose launch fails
void fake_clear() { g_launches.clear(); }
int fake_count() { return (int)g_launches.size(); }
const char* fake_name(int i) { return g_launches[i].c_str(); }

// ---- registration and launches, as compiled host code calls them
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
static size_t g_cfg_smem;
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t smem, cudaStream_t) { g_cfg_smem = smem; return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t* smem, void*) { *smem = g_cfg_smem; return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t smem, cudaStream_t) {
  return launch((const void*)k, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (!g_refuse.empty() && g_names[f].find(g_refuse) != std::string::npos) return set(cudaErrorInvalidValue);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (v > 227 * 1024) return set(cudaErrorInvalidValue);
    g_smem[{g_dev, f}] = (size_t)v;
  }
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return g_last; }
const char* cudaGetErrorString(cudaError_t) { return "error of the host runtime"; }

// ---- devices and memory
cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeDevice;
  a->device = g_dev;
  a->devicePointer = const_cast<void*>(p);
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return (*p = calloc(n, 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t n) {
  double* d = (double*)malloc(n + 8);
  for (size_t i = 0; i <= n / 8; ++i) d[i] = 1.0;
  *p = d;
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { *d = h; return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { memmove(d, s, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { memset(d, v, n); return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { *p = const_cast<void*>(s); return cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = (void*)encode_tiled;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamGetDevice(cudaStream_t, int* d) { *d = g_dev; return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventQuery(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 0.f; return cudaSuccess; }
}
