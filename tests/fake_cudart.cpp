// A CUDA runtime for tests of the host code on machines without a GPU: device
// memory is host memory, kernels do not run, and every kernel launch and
// memset is recorded.  As on a device, the dynamic shared memory of a kernel
// above 48 KB has to be allowed first, on each device by itself.  A launch of
// a kernel whose name holds a given text can be made to fail.  Linked with the
// library's objects in place of the CUDA runtime; the functions keep the names
// and signatures of the runtime's headers.
#include <cuda_runtime_api.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <string>
#include <vector>

namespace {
struct Event {
  int kind;            // 0 kernel, 1 memset, 2 refused or failed kernel
  std::string name;    // kernel
  size_t bytes;        // memset
};
int g_device = 0;
cudaError_t g_last = cudaSuccess;
std::map<const void*, std::string> g_names;
std::map<std::pair<int, const void*>, size_t> g_smem;
std::vector<Event> g_log;
std::string g_fail;
int g_fail_left = 0;
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} g_config;
cudaError_t result(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}
int encode_tiled(void*, ...) { return 0; }
}  // namespace

extern "C" {
#define FAKE __attribute__((visibility("default")))

// ---- controls of the tests
FAKE void fake_set_device(int d) { g_device = d; }
FAKE void fake_clear() {
  g_log.clear();
  g_last = cudaSuccess;
  g_fail_left = 0;
}
FAKE void fake_fail(const char* name, int times) {
  g_fail = name;
  g_fail_left = times;
}
FAKE int fake_count() { return (int)g_log.size(); }
FAKE int fake_kind(int i) { return g_log[i].kind; }
FAKE const char* fake_name(int i) { return g_log[i].name.c_str(); }
FAKE long fake_bytes(int i) { return (long)g_log[i].bytes; }

// ---- what the compiler's launch code calls
void** __cudaRegisterFatBinary(void*) {
  static void* h[1];
  return h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* fun, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_names[fun] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* s) {
  g_config = {grid, block, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  *grid = g_config.grid;
  *block = g_config.block;
  *smem = g_config.smem;
  *static_cast<cudaStream_t*>(s) = g_config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fun) {
  *k = (cudaKernel_t)fun;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t smem, cudaStream_t) {
  const void* fun = (const void*)k;
  const std::string& name = g_names[fun];
  const unsigned threads = block.x * block.y * block.z;
  const auto allowed = g_smem.find({g_device, fun});
  cudaError_t e = cudaSuccess;
  if (grid.x == 0 || grid.y == 0 || grid.z == 0 || threads == 0 || threads > 1024) e = cudaErrorInvalidConfiguration;
  if (smem > 48 * 1024 && (allowed == g_smem.end() || allowed->second < smem)) e = cudaErrorInvalidValue;
  if (g_fail_left > 0 && name.find(g_fail) != std::string::npos) {
    --g_fail_left;
    e = cudaErrorMemoryAllocation;   // as the first use of a kernel on a full device
  }
  g_log.push_back({e == cudaSuccess ? 0 : 2, name, 0});
  return result(e);
}

// ---- the runtime
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return g_last; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "error of the fake runtime"; }
cudaError_t cudaGetDevice(int* d) {
  *d = g_device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* fun, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (v > 227 * 1024) return result(cudaErrorInvalidValue);
    g_smem[{g_device, fun}] = (size_t)v;
  }
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int threads, size_t smem) {
  const int by_smem = (int)(227 * 1024 / (smem + 1024)), by_threads = 2048 / threads;
  *n = by_smem < by_threads ? by_smem : by_threads;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int threads, size_t smem,
                                                                   unsigned) {
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, f, threads, smem);
}
cudaError_t cudaMalloc(void** p, size_t bytes) {
  *p = calloc(1, bytes);
  return *p ? cudaSuccess : result(cudaErrorMemoryAllocation);
}
cudaError_t cudaFree(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t bytes) { return cudaMalloc(p, bytes); }
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemset(void*, int, size_t bytes) {
  g_log.push_back({1, "", bytes});
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t bytes, cudaStream_t) { return cudaMemset(p, v, bytes); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t bytes, cudaMemcpyKind) {
  memcpy(d, s, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t bytes, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, bytes, k);
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static char room[1 << 24];
  *p = room;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *fn = (void*)&encode_tiled;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)calloc(1, 16);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  free(s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamGetDevice(cudaStream_t, int* d) { return cudaGetDevice(d); }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return result(cudaErrorNotSupported); }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return result(cudaErrorNotSupported); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return result(cudaErrorNotSupported); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return result(cudaErrorNotSupported); }
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t*) { return result(cudaErrorNotSupported); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t)calloc(1, 16);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  free(e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.0f;
  return cudaSuccess;
}
}  // extern "C"
