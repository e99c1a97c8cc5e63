// A stand-in for the CUDA runtime, linked into the library's host code by test_launch_chain.py: it keeps the dynamic
// shared-memory limit of every kernel as the runtime does (one per function, the last call decides), refuses a launch
// above it, or one the test asks it to refuse, and writes down which kernels were launched.  No kernel ever runs.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
std::map<const void*, size_t>& limits() {
  static std::map<const void*, size_t> m;
  return m;
}
std::vector<std::string> launched;
int refuse_at = -1, asked = 0;
cudaError_t last = cudaSuccess;
bool capturing = false;
void* host_memory = nullptr;   // the last pinned allocation

cudaError_t launch(const void* func, size_t smem) {
  const size_t limit = limits().count(func) ? limits()[func] : 48 * 1024;
  if (asked++ == refuse_at || smem > limit) return last = cudaErrorInvalidValue;
  launched.push_back(names()[func]);
  return cudaSuccess;
}
CUresult encode_tiled(CUtensorMap*, ...) { return CUDA_SUCCESS; }
}  // namespace

extern "C" {
// ---- for the test
void fake_reset(int refuse) {
  launched.clear();
  asked = 0;
  refuse_at = refuse;
}
int fake_launched() { return (int)launched.size(); }
const char* fake_name(int i) { return launched[i].c_str(); }
void fake_capturing(int on) { capturing = on != 0; }
void* fake_host_memory() { return host_memory; }

// ---- what the compiler's registration code calls
void** __cudaRegisterFatBinary(void*) {
  static void* handle;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
char __cudaInitModule(void**) { return 0; }
void __cudaRegisterFunction(void**, const char* func, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) { names()[func] = name; }
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
static dim3 g_grid, g_block;
static size_t g_smem;
static void* g_stream;
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, void* stream) {
  g_grid = grid;
  g_block = block;
  g_smem = smem;
  g_stream = stream;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = g_grid;
  *block = g_block;
  *smem = g_smem;
  *(void**)stream = g_stream;
  return cudaSuccess;
}

// ---- the runtime
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t smem, cudaStream_t) { return launch(f, smem); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->dynamicSmemBytes); }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute attr, int value) {
  if (attr == cudaFuncAttributeMaxDynamicSharedMemorySize) limits()[f] = (size_t)value;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {   // cudaGetDeviceProperties_v2 by the header's macro
  memset(p, 0, sizeof(*p));
  p->major = 10;
  p->multiProcessorCount = 148;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** p, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *p = (void*)encode_tiled;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { return *n = 74, cudaSuccess; }
cudaError_t cudaMalloc(void** p, size_t n) { return *p = malloc(n), cudaSuccess; }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { return *p = (void*)s, cudaSuccess; }
cudaError_t cudaMemcpy(void*, const void*, size_t, cudaMemcpyKind) { return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return host_memory = *p = calloc(1, n), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) {
  if (p == host_memory) host_memory = nullptr;
  return free(p), cudaSuccess;
}
cudaError_t cudaStreamQuery(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t*, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t*) { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t*, unsigned) { return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 0.f, cudaSuccess; }
}
