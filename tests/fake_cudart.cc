#include "fake_cudart.h"

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>

namespace fake {

std::map<void*, size_t> live;
std::map<std::string, int> launched;
std::function<void(const std::string&, void**)> on_launch;
std::function<void(void*, size_t)> on_copy;
int64_t allocs = 0, fail_from = -1, fail_count = 0;
size_t used = 0, peak = 0, capacity = SIZE_MAX;
bool no_streams = false;
int graph_launches = 0, graphs = 0;

[[noreturn]] void die(const char* fmt, ...) {
  va_list a;
  va_start(a, fmt);
  vfprintf(stderr, fmt, a);
  va_end(a);
  fputc('\n', stderr);
  exit(2);
}

std::map<const void*, std::string>& names() {  // kernels by host entry
  static std::map<const void*, std::string> m;
  return m;
}

void launch(const void* f, void** args) {
  const auto it = names().find(f);
  if (it == names().end()) die("launch of an unknown kernel");
  launched[it->second]++;
  if (on_launch) on_launch(it->second, args);
}

bool named(const std::string& mangled, const char* kernel) { return mangled.find(kernel) != std::string::npos; }

int launches(const char* kernel) {
  int n = 0;
  for (const auto& [name, count] : launched) n += named(name, kernel) ? count : 0;
  return n;
}

void need(const char* what, const void* p, size_t bytes) {
  const auto it = live.find(const_cast<void*>(p));
  if (it == live.end()) die("%s: %p is not allocated", what, p);
  if (it->second < bytes) die("%s: %zu bytes, %zu needed", what, it->second, bytes);
}

int plain_handle;


}  // namespace fake

struct dim3_config {
  dim3 grid, block;
  size_t smem;
  void* stream;
};
static dim3_config g_config;

extern "C" {
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&fake::plain_handle); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  fake::names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* stream) {
  g_config = {grid, block, smem, stream};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* stream) {
  *grid = g_config.grid;
  *block = g_config.block;
  *smem = g_config.smem;
  *static_cast<void**>(stream) = g_config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* entry) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(entry));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t, cudaStream_t) {
  fake::launch(k, args);
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* f, void** args) {
  fake::launch(f, args);
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t bytes, cudaStream_t) {
  const int64_t n = fake::allocs++;
  *p = nullptr;
  if ((fake::fail_from >= 0 && n >= fake::fail_from && n < fake::fail_from + fake::fail_count) ||
      fake::used + bytes > fake::capacity)
    return cudaErrorMemoryAllocation;
  *p = calloc(bytes, 1);
  fake::live[*p] = bytes;
  fake::used += bytes;
  fake::peak = std::max(fake::peak, fake::used);
  return cudaSuccess;
}
cudaError_t cudaFreeAsync(void* p, cudaStream_t) {
  if (!p) return cudaSuccess;
  const auto it = fake::live.find(p);
  if (it == fake::live.end()) fake::die("freed what is not allocated: %p", p);
  fake::used -= it->second;
  fake::live.erase(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t bytes) { return (*p = calloc(bytes, 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaMemcpyAsync(void* to, const void* from, size_t bytes, cudaMemcpyKind, cudaStream_t) {
  if (bytes && (!to || !from)) fake::die("copy of %zu bytes from %p to %p", bytes, from, to);
  if (bytes) memmove(to, from, bytes);
  if (fake::on_copy) fake::on_copy(to, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* to, const void* from, size_t bytes, cudaMemcpyKind) {
  if (bytes && (!to || !from)) return cudaErrorInvalidValue;
  if (bytes) memmove(to, from, bytes);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t bytes, cudaStream_t) {
  if (bytes && !p) fake::die("fill of %zu bytes at null", bytes);
  if (bytes) memset(p, v, bytes);
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaDeviceGetDefaultMemPool(cudaMemPool_t*, int) { return cudaErrorNotSupported; }
cudaError_t cudaMemPoolSetAttribute(cudaMemPool_t, cudaMemPoolAttr, void*) { return cudaSuccess; }
static int g_objects;
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = reinterpret_cast<cudaEvent_t>(&g_objects), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* t, cudaEvent_t, cudaEvent_t) { return *t = 0.f, cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidSymbol; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* g, cudaGraph_t, unsigned long long) {
  fake::graphs++;
  return *g = reinterpret_cast<cudaGraphExec_t>(&g_objects), cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return fake::graph_launches++, cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* b, const void*, int, size_t, unsigned) {
  return *b = 1, cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) { return *a = {}, cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return *g = reinterpret_cast<cudaGraph_t>(&g_objects), cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  if (fake::no_streams) return *s = nullptr, cudaErrorMemoryAllocation;
  return *s = reinterpret_cast<cudaStream_t>(&g_objects), cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
}
