// A CUDA runtime without a device, for tests of the library's host code: the
// library's own object files are linked against it instead of the CUDA runtime.
// Kernels do not run.  Each launch is recorded with the launches that stream
// order and events put before it, so a test can ask whether one kernel waits for
// another.  Memory is host memory; copies take place at once.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

namespace {
struct Launch {
  std::string name;
  std::set<int> before;   // launches ordered before this one
};
std::map<const void*, std::string>& names() {   // filled while the library loads
  static std::map<const void*, std::string> n;
  return n;
}
std::vector<Launch> launches;
std::map<void*, std::set<int>> done;   // launches that have ended where a stream or an event stands
struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} config;
uintptr_t next_handle = 16;
int host_allocs = 0, device_allocs = 0;   // page-locked blocks held, device allocations since the reset
template <class T>
cudaError_t make(T* h) {
  *h = reinterpret_cast<T>(next_handle += 16);
  return cudaSuccess;
}
cudaError_t alloc(void** p, size_t n) {
  *p = aligned_alloc(256, (n + 511) / 256 * 256);
  if (!*p) return cudaErrorMemoryAllocation;
  std::memset(*p, 0, n);
  return cudaSuccess;
}
CUresult encode_tiled(CUtensorMap* m, ...) {
  std::memset(m, 0, sizeof *m);
  return CUDA_SUCCESS;
}
}  // namespace

extern "C" {
// ---- what a test asks
void fake_reset() { launches.clear(), done.clear(), device_allocs = 0; }
int fake_host_allocs() { return host_allocs; }
int fake_device_allocs() { return device_allocs; }
int fake_count() { return (int)launches.size(); }
const char* fake_name(int i) { return launches[i].name.c_str(); }
int fake_before(int a, int b) { return (int)launches[b].before.count(a); }

// ---- registration and launches
void** __cudaRegisterFatBinary(void*) { return nullptr; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, cudaStream_t s) {
  config = {g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = config.grid, *b = config.block, *smem = config.smem;
  *static_cast<cudaStream_t*>(s) = config.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t s) {
  std::set<int>& at = done[s];
  launches.push_back({names()[(const void*)k], at});
  at.insert((int)launches.size() - 1);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  done[e] = done[s];
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  const std::set<int> at = done[e];
  done[s].insert(at.begin(), at.end());
  return cudaSuccess;
}

// ---- the rest succeeds
cudaError_t cudaMalloc(void** p, size_t n) { return ++device_allocs, alloc(p, n); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return ++host_allocs, alloc(p, n); }
cudaError_t cudaFree(void* p) { return free(p), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return --host_allocs, free(p), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) { return std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* s) { return *p = const_cast<void*>(s), cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return make(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return make(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.0f, cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return make(s); }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return make(g); }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { return make(x); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  return *n = 2, cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = (void*)&encode_tiled;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
}
