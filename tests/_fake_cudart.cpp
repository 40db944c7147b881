// A CUDA runtime that runs nothing, for tests of the library's host side: device
// memory is host memory, launches are recorded (with the name their kernel was
// registered under) and never executed, and time is the cost of what was launched.
// Linked with the library's objects in place of the real runtime.
#include <cuda_runtime_api.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

namespace {
int g_device = 0;
std::map<const void*, std::string> g_name;                    // kernel -> registered name
std::map<std::pair<const void*, int>, int> g_smem;            // (kernel, device) -> allowed bytes
struct Launch {
  const void* func;
  int device, grid_x, grid_y, smem, refused;
};
std::vector<Launch> g_launch;
std::string g_fast;   // kernels whose name contains this cost 1, others 10
double g_clock = 0.0;
std::map<cudaEvent_t, double> g_event;
uintptr_t g_next = 0x1000;

cudaError_t launch(const void* f, dim3 grid, size_t smem) {
  const auto it = g_smem.find({f, g_device});
  const int allowed = it == g_smem.end() ? 48 * 1024 : it->second;
  g_launch.push_back({f, g_device, (int)grid.x, (int)grid.y, (int)smem, (int)smem > allowed});
  g_clock += !g_fast.empty() && g_name[f].find(g_fast) != std::string::npos ? 1.0 : 10.0;
  return g_launch.back().refused ? cudaErrorInvalidValue : cudaSuccess;
}
int encode(...) { return 0; }
}  // namespace

extern "C" {
// The test's side.
void fake_set_device(int d) { g_device = d; }
void fake_set_fast(const char* s) { g_fast = s; }
int fake_launches() { return (int)g_launch.size(); }
const char* fake_launch(int i, int* device, int* grid_x, int* grid_y, int* smem) {
  const Launch& l = g_launch[i];
  *device = l.device, *grid_x = l.grid_x, *grid_y = l.grid_y, *smem = l.smem;
  return g_name[l.func].c_str();
}

// What the library and the compiler's registration code call.
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&g_next); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  g_name[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void**, size_t smem, cudaStream_t) {
  return launch((const void*)k, grid, smem);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(f, c->gridDim, c->dynamicSmemBytes);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int v) {
  g_smem[{f, g_device}] = v;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t,
                                                                   unsigned) {
  *n = 4;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = g_device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *f = reinterpret_cast<void*>(&encode);
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = std::calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  std::memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static double words[4096];
  *p = words;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "fake runtime"; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  *e = (cudaEvent_t)(g_next += 16);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
  g_event[e] = g_clock;
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = (float)(g_event[b] - g_event[a]);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)(g_next += 16);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
// Only batches with a stream of their own capture graphs; the tests give none.
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaErrorNotSupported; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t*) { return cudaErrorNotSupported; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t*, cudaGraph_t, unsigned long long) { return cudaErrorNotSupported; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaErrorNotSupported; }
}
