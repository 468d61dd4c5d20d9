// A stand-in for the CUDA runtime, for tests of the library's host side without a GPU.
//
// Loaded before the library (LD_PRELOAD, see fake_cuda.py) it answers the runtime calls the
// library makes: device memory is host memory, copies happen at once, kernels do not run.
// Launches, shared memory limits, copies to the host and synchronisations go to a log; a
// launch advances its stream's clock by a time the test chooses, which events read; any
// call can be made to fail.
#include <cuda_runtime_api.h>
#include <cxxabi.h>
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <map>
#include <mutex>
#include <string>
#include <vector>

namespace {

std::recursive_mutex mu;
std::string log_, taken;
std::map<const void*, std::string> names;  // kernels by their host address
std::map<std::string, int> failing;        // calls left before a function fails once
struct Cost {
  std::string kernel;
  unsigned grid, block;
  float us;
};
std::vector<Cost> costs;
std::map<std::string, int> resident;
std::map<std::string, unsigned> watched;  // byte of a kernel's first argument at which a word is logged
std::map<uintptr_t, double> clocks;  // us, by stream
uintptr_t handles = 0x1000;
struct Launch {
  dim3 grid, block;
  size_t smem;
  void* stream;
};
thread_local std::vector<Launch> pushed;

void note(const char* fmt, ...) {
  char b[2048];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(b, sizeof b, fmt, ap);
  va_end(ap);
  std::lock_guard<std::recursive_mutex> g(mu);
  log_ += b;
  log_ += '\n';
}

bool fails(const char* fn) {
  std::lock_guard<std::recursive_mutex> g(mu);
  auto it = failing.find(fn);
  if (it == failing.end()) return false;
  if (it->second-- > 0) return false;
  failing.erase(it);
  note("failed %s", fn);
  return true;
}
#define FAIL(fn) \
  if (fails(#fn)) return cudaErrorUnknown

std::string name_of(const void* f) {
  std::lock_guard<std::recursive_mutex> g(mu);
  auto it = names.find(f);
  return it == names.end() ? "?" : it->second;
}

cudaError_t launch(const void* f, dim3 g, dim3 b, size_t smem, void* s) {
  const std::string n = name_of(f);
  std::lock_guard<std::recursive_mutex> lock(mu);
  note("launch %lu %u %u %zu %s", (unsigned long)(uintptr_t)s, g.x * g.y * g.z, b.x, smem, n.c_str());
  double us = 10.0;
  for (const Cost& c : costs)
    if (n.find(c.kernel) != std::string::npos && c.grid == g.x * g.y * g.z && c.block == b.x) us = c.us;
  clocks[(uintptr_t)s] += us;
  return cudaSuccess;
}

void* handle() { return (void*)(handles += 16); }

}  // namespace

extern "C" {

// ---- the test's side
const char* fake_take_log() {
  std::lock_guard<std::recursive_mutex> g(mu);
  taken.swap(log_);
  log_.clear();
  return taken.c_str();
}
void fake_fail(const char* fn, int after) {  // the call after `after` more of them fails
  std::lock_guard<std::recursive_mutex> g(mu);
  failing[fn] = after;
}
void fake_cost(const char* kernel, unsigned grid, unsigned block, float us) {
  std::lock_guard<std::recursive_mutex> g(mu);
  costs.push_back(Cost{kernel, grid, block, us});
}
void fake_resident(const char* kernel, int per_sm) {
  std::lock_guard<std::recursive_mutex> g(mu);
  resident[kernel] = per_sm;
}

void fake_watch(const char* kernel, unsigned offset) { watched[kernel] = offset; }

// ---- the library's side
void** __cudaRegisterFatBinary(void*) { return (void**)handle(); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* device, int, uint3*, uint3*, dim3*, dim3*,
                            int*) {
  int st = 0;
  char* d = abi::__cxa_demangle(device, NULL, NULL, &st);
  std::lock_guard<std::recursive_mutex> g(mu);
  names[host] = st == 0 ? d : device;
  free(d);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, void* s) {
  pushed.push_back(Launch{g, b, smem, s});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  const Launch l = pushed.back();
  pushed.pop_back();
  *g = l.grid;
  *b = l.block;
  *smem = l.smem;
  *(void**)s = l.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t s) {
  return launch((const void*)k, g, b, smem, s);
}
cudaError_t cudaLaunchKernel(const void* f, dim3 g, dim3 b, void**, size_t smem, cudaStream_t s) {
  return launch(f, g, b, smem, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  FAIL(cudaLaunchKernelExC);
  const std::string n = name_of(f);
  for (const auto& w : watched)
    if (n.find(w.first) != std::string::npos) note("word %d", *(const int*)((const char*)args[0] + w.second));
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  FAIL(cudaFuncSetAttribute);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) note("limit %d %s", v, name_of(f).c_str());
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void* f, int, size_t, unsigned) {
  const std::string k = name_of(f);
  std::lock_guard<std::recursive_mutex> g(mu);
  *n = 1;
  for (const auto& r : resident)
    if (k.find(r.first) != std::string::npos) *n = r.second;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  FAIL(cudaMalloc);
  *p = aligned_alloc(256, (n + 255) / 256 * 256);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  FAIL(cudaMemcpyAsync);
  memcpy(d, s, n);
  if (k == cudaMemcpyDeviceToHost) note("d2h %lu %zu", (unsigned long)(uintptr_t)st, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  FAIL(cudaMemcpy);
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  FAIL(cudaMemsetAsync);
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  memset(d, v, n);
  return cudaSuccess;
}
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)handle();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  note("destroy %lu", (unsigned long)(uintptr_t)s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  note("sync %lu", (unsigned long)(uintptr_t)s);
  FAIL(cudaStreamSynchronize);
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) {
  FAIL(cudaStreamWaitEvent);
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = (cudaGraph_t)handle();
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = (cudaGraphExec_t)handle();
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t) new double(0);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  delete (double*)e;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  FAIL(cudaEventRecord);
  std::lock_guard<std::recursive_mutex> g(mu);
  *(double*)e = clocks[(uintptr_t)s];
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = (float)((*(double*)b - *(double*)a) * 1e-3);
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : (a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0);
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "stand-in error"; }
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorUnknown; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void**, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult*) {
  return cudaErrorUnknown;
}

}  // extern "C"
