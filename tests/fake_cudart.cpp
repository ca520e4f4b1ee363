// A CUDA runtime without a GPU, to link the library's objects against on the CPU:
// device memory is host memory, copies and fills are done, kernels are not run. The
// launch number fake_fail_at (from 1 on; 0: none) is refused as the runtime refuses a
// launch: an error code, kept for cudaGetLastError.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <atomic>
#include <cstdlib>
#include <cstring>

extern "C" {
std::atomic<long long> fake_launches{0}, fake_fail_at{0};
}

namespace {
thread_local cudaError_t g_last = cudaSuccess;  // as the runtime's: per host thread
struct Config {
  dim3 grid, block;
  size_t smem;
  void* stream;
};
thread_local Config g_config;
char g_handle;

cudaError_t launch() {
  if (++fake_launches != fake_fail_at) return cudaSuccess;
  return g_last = cudaErrorInvalidConfiguration;
}
cudaError_t alloc(void** p, size_t n) {
  *p = std::calloc(n ? n : 1, 1);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
CUresult encode(CUtensorMap*) { return CUDA_SUCCESS; }
}  // namespace

extern "C" {
#define OK(name, ...) \
  cudaError_t name(__VA_ARGS__) { return cudaSuccess; }

unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
  g_config = Config{grid, block, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = g_config.grid;
  *block = g_config.block;
  *smem = g_config.smem;
  *static_cast<void**>(stream) = g_config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void*) {
  *k = nullptr;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) {
  return launch();
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return launch(); }
cudaError_t cudaLaunchCooperativeKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) {
  return launch();
}
void** __cudaRegisterFatBinary(void*) {
  static void* handle = nullptr;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*,
                            dim3*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "fake"; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
OK(cudaSetDevice, int)
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t,
                                                                   unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) { return alloc(p, n); }
cudaError_t cudaMallocHost(void** p, size_t n) { return alloc(p, n); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return alloc(p, n); }
cudaError_t cudaFree(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t pd, const void* s, size_t ps, size_t w, size_t h,
                              cudaMemcpyKind, cudaStream_t) {
  for (size_t i = 0; i < h; ++i)
    std::memmove(static_cast<char*>(d) + i * pd, static_cast<const char*>(s) + i * ps, w);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return cudaMemset(d, v, n); }
cudaError_t cudaMemset2DAsync(void* d, size_t pitch, int v, size_t w, size_t h, cudaStream_t) {
  for (size_t i = 0; i < h; ++i) std::memset(static_cast<char*>(d) + i * pitch, v, w);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return alloc(p, 1 << 22); }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(&g_handle);
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.f;
  return cudaSuccess;
}
OK(cudaEventDestroy, cudaEvent_t)
OK(cudaEventRecord, cudaEvent_t, cudaStream_t)
OK(cudaEventSynchronize, cudaEvent_t)
OK(cudaFuncSetAttribute, const void*, cudaFuncAttribute, int)
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(&g_handle);
  return cudaSuccess;
}
OK(cudaStreamDestroy, cudaStream_t)
OK(cudaStreamSynchronize, cudaStream_t)
OK(cudaStreamBeginCapture, cudaStream_t, cudaStreamCaptureMode)
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = reinterpret_cast<cudaGraph_t>(&g_handle);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  *x = reinterpret_cast<cudaGraphExec_t>(&g_handle);
  return cudaSuccess;
}
OK(cudaGraphDestroy, cudaGraph_t)
OK(cudaGraphExecDestroy, cudaGraphExec_t)
OK(cudaGraphLaunch, cudaGraphExec_t, cudaStream_t)
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *fn = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}
