// A CUDA runtime for host tests: linked with the library's objects in place of
// libcudart.  Device memory is host memory counted against a budget, kernels do
// not run (their launches are logged), streams run at once, and any call can be
// told to return an error.  Only what the library calls is here.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>

namespace {

std::mutex mu;
std::map<void*, size_t> blocks;
size_t live = 0, peak = 0, budget = 0;
std::map<std::string, std::pair<int, int>> failing;  // call -> (calls until it fails, error)
std::map<const void*, std::string> names;
std::string launches;
bool capturing = false;
int graph_launches = 0;  // since the last cudaEventElapsedTime
float graph_ms = 1.f;
cudaError_t last = cudaSuccess;
thread_local dim3 cfg_grid, cfg_block;
thread_local size_t cfg_smem;
thread_local cudaStream_t cfg_stream;
char token;

cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) last = e;
  return e;
}
cudaError_t result(const char* call) {
  auto it = failing.find(call);
  if (it == failing.end() || --it->second.first > 0) return cudaSuccess;
  const int code = it->second.second;
  failing.erase(it);
  return set((cudaError_t)code);
}

}  // namespace

extern "C" {

// ---- control ------------------------------------------------------------
void fake_reset() {
  std::lock_guard<std::mutex> l(mu);
  failing.clear();
  launches.clear();
  budget = 0;
  peak = live;
  last = cudaSuccess;
  graph_launches = 0;
  graph_ms = 1.f;
}
void fake_budget(size_t bytes) { budget = bytes; }  // 0 = no limit
size_t fake_live() { return live; }
size_t fake_peak() { return peak; }
void fake_fail(const char* call, int nth, int code) { failing[call] = {nth, code}; }
const char* fake_launches() { return launches.c_str(); }  // "kernel grid block smem captured" a line

// ---- launches -------------------------------------------------------------
void** __cudaRegisterFatBinary(void*) { return reinterpret_cast<void**>(&token); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  cfg_grid = g;
  cfg_block = b;
  cfg_smem = smem;
  cfg_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = cfg_grid;
  *b = cfg_block;
  *smem = cfg_smem;
  *static_cast<cudaStream_t*>(s) = cfg_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t) {
  std::lock_guard<std::mutex> l(mu);
  auto d = [](dim3 v) { return std::to_string(v.x) + "," + std::to_string(v.y) + "," + std::to_string(v.z); };
  launches += names[k] + " " + d(g) + " " + d(b) + " " + std::to_string(smem) + (capturing ? " 1\n" : " 0\n");
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}

// ---- memory ---------------------------------------------------------------
cudaError_t cudaMalloc(void** p, size_t n) {
  std::lock_guard<std::mutex> l(mu);
  cudaError_t e = result("cudaMalloc");
  if (e == cudaSuccess && budget && live + n > budget) e = set(cudaErrorMemoryAllocation);
  if (e != cudaSuccess) return e;
  *p = calloc(n ? n : 1, 1);
  blocks[*p] = n;
  live += n;
  if (live > peak) peak = live;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  std::lock_guard<std::mutex> l(mu);
  if (!p) return cudaSuccess;
  auto it = blocks.find(p);
  if (it == blocks.end()) return set(cudaErrorInvalidValue);
  live -= it->second;
  blocks.erase(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
  if (!p) return set(cudaErrorInvalidValue);
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  return capturing ? cudaSuccess : cudaMemset(p, v, n);
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  if (!d || !s) return set(cudaErrorInvalidValue);
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return capturing ? cudaSuccess : cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t, const void* s, size_t, size_t, size_t, cudaMemcpyKind, cudaStream_t) {
  return d && s ? cudaSuccess : set(cudaErrorInvalidValue);
}
cudaError_t cudaMemcpy3DAsync(const cudaMemcpy3DParms* p, cudaStream_t) {
  return p->srcPtr.ptr && p->dstPtr.ptr ? cudaSuccess : set(cudaErrorInvalidValue);
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static void* block = calloc(64u << 20, 1);
  *p = block;
  return cudaSuccess;
}
// every host address counts as page-locked
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  *a = cudaPointerAttributes{};
  a->type = cudaMemoryTypeHost;
  a->devicePointer = a->hostPointer = const_cast<void*>(p);
  return cudaSuccess;
}

// ---- device, errors ---------------------------------------------------------
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = last;
  last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "planted error"; }

// ---- streams, events, graphs -------------------------------------------------
cudaError_t cudaStreamSynchronize(cudaStream_t) { return result("cudaStreamSynchronize"); }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(&token);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  capturing = true;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  capturing = false;
  *g = reinterpret_cast<cudaGraph_t>(&token);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  const cudaError_t r = result("cudaGraphInstantiate");
  if (r == cudaSuccess) *e = reinterpret_cast<cudaGraphExec_t>(&token);
  return r;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  ++graph_launches;
  return result("cudaGraphLaunch");
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(&token);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  // a graph takes 10 % less each time, so that a tuner keeps the last of its
  // candidates; all other launches take the same
  *ms = graph_launches ? graph_ms *= 0.9f : 1.f;
  graph_launches = 0;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }

}  // extern "C"
