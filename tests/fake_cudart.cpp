// A CUDA runtime without a device, for tests of the library's host code: streams, events,
// copies and launches are only written down, memory is a range of addresses behind which
// there is nothing, and chosen calls fail. Loaded before libhv.so, whose calls then come here.
#include <cuda_runtime_api.h>

#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

#include "hv_internal.h"

namespace {
std::string g_log, g_out;
std::map<size_t, size_t> g_live;  // address -> bytes
std::map<const void*, std::string> g_name;
size_t g_next = size_t(1) << 32, g_fail_from = 0, g_fail_to = 0;
int g_fail_malloc = 0, g_fail_launch = 0;
std::string g_fail_kernel;
cudaError_t g_last = cudaSuccess;
size_t g_handle = 16;
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
};
std::vector<Config> g_config;

void log(const char* fmt, ...) __attribute__((format(printf, 1, 2)));
void log(const char* fmt, ...) {
  char line[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(line, sizeof(line), fmt, ap);
  va_end(ap);
  g_log += line;
  g_log += '\n';
}
size_t num(const void* p) { return reinterpret_cast<size_t>(p); }
cudaError_t err(cudaError_t e) { return g_last = e; }

// Bytes of the live allocation from p on, 0 outside.
size_t room(const void* p) {
  auto it = g_live.upper_bound(num(p));
  if (it == g_live.begin()) return 0;
  --it;
  return num(p) < it->first + it->second ? it->first + it->second - num(p) : 0;
}

cudaError_t launch(const void* f, void** args, cudaStream_t s) {
  const std::string name = g_name.count(f) ? g_name[f] : "?";
  if (g_fail_launch > 0 && name.find(g_fail_kernel) != std::string::npos) {
    --g_fail_launch;
    return err(cudaErrorLaunchFailure);
  }
  log("kernel %zu %s", num(s), name.c_str());
  if (name.find("k_strip_") != std::string::npos || name.find("k_feature_pass") != std::string::npos) {
    const hv::SpatialArgs& a = *static_cast<const hv::SpatialArgs*>(args[0]);
    log("scratch %u %u %u %d %zu %zu", a.W, a.H, a.n, a.spatial, room(a.scratch1), room(a.scratch2));
  }
  return cudaSuccess;
}
int encode(...) { return 0; }  // cuTensorMapEncodeTiled
}  // namespace

extern "C" {
const char* fake_log() {
  g_out.swap(g_log);
  g_log.clear();
  return g_out.c_str();
}
// The next `times` allocations of `from` to `to` bytes fail.
void fake_fail_malloc(size_t from, size_t to, int times) { g_fail_from = from, g_fail_to = to, g_fail_malloc = times; }
// The next `times` launches of a kernel whose name holds `part` fail.
void fake_fail_launch(const char* part, int times) { g_fail_kernel = part, g_fail_launch = times; }

cudaError_t cudaMalloc(void** p, size_t n) {
  *p = nullptr;
  if (g_fail_malloc > 0 && n >= g_fail_from && n <= g_fail_to) {
    --g_fail_malloc;
    return err(cudaErrorMemoryAllocation);
  }
  *p = reinterpret_cast<void*>(g_next);
  g_live[g_next] = n;
  log("malloc %zu %zu", g_next, n);
  g_next += (n + 4095) / 4096 * 4096 + 4096;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (p && !g_live.erase(num(p))) return err(cudaErrorInvalidValue);
  log("free %zu", num(p));
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void*, size_t n, cudaMemcpyKind k) {
  log("sync");
  if (k == cudaMemcpyDeviceToHost) memset(d, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  log("copy %zu %zu %zu %zu", num(st), num(d), num(s), n);
  if (k == cudaMemcpyDeviceToHost) memset(d, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) {
  log("sync");
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return *p = malloc(n), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return free(p), cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(g_handle += 16);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) { return log("host_stream %zu", num(s)), cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  return log("wait %zu %zu", num(s), num(e)), cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) { return log("capture %zu", num(s)), cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  *g = reinterpret_cast<cudaGraph_t>(g_handle += 16);
  return log("end %zu", num(s)), cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) {
  *x = reinterpret_cast<cudaGraphExec_t>(g_handle += 16);
  return cudaSuccess;
}
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t, cudaGraph_t, cudaGraphExecUpdateResultInfo*) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) { return log("graph %zu", num(s)), cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }

cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) {
  *e = reinterpret_cast<cudaEvent_t>(g_handle += 16);
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return cudaEventCreateWithFlags(e, 0); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return log("record %zu %zu", num(s), num(e)), cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t e) { return log("host_event %zu", num(e)), cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }

cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  *a = cudaFuncAttributes{};
  a->numRegs = 64;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 2, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { return *n = 4, cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return cudaMalloc(p, 4096); }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return g_last; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }

cudaError_t __cudaGetKernel(const void** k, const void* f) { return *k = f, cudaSuccess; }
cudaError_t __cudaLaunchKernel(const void* f, dim3, dim3, void** args, size_t, cudaStream_t s) { return launch(f, args, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) { return launch(f, args, c->stream); }
cudaError_t cudaLaunchCooperativeKernel(const void* f, dim3, dim3, void** args, size_t, cudaStream_t s) {
  return launch(f, args, s);
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t m, void* s) {
  g_config.push_back(Config{g, b, m, static_cast<cudaStream_t>(s)});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* m, void* s) {
  const Config c = g_config.back();
  g_config.pop_back();
  *g = c.grid, *b = c.block, *m = c.smem, *static_cast<cudaStream_t*>(s) = c.stream;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void* f) { return static_cast<void**>(f); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  g_name[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
