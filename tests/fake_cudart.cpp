// A stand-in for the CUDA runtime, for tests of the library's host code on a machine without a GPU
// (tests/test_host_paths.py): device memory is host memory, kernels do not run, and every launch is
// held against the limits and the allocations that a device would hold it against.
//   - cudaFuncSetAttribute holds for the current device alone, as the runtime documents it; a launch
//     with more dynamic shared memory than its kernel's limit there (48 KiB unless raised) fails.
//   - fake_fail_alloc(i): the allocation after the next i ones fails; fake_limit(b): those that would
//     take the total above b bytes; fake_fail_attr(1): every cudaFuncSetAttribute.
//   - fake_watch(name, arg): the pointer argument `arg` of every launch of a kernel whose name
//     contains `name` has to lie inside a live allocation; fake_bad() counts those that do not.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <limits>
#include <map>
#include <string>
#include <utility>
#include <vector>

namespace {

struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t st;
};

int g_device = 0, g_fail_attr = 0;
long long g_fail_alloc = -1, g_byte_limit = -1;
long long g_bad = 0, g_reads = 0, g_launches = 0, g_graph_launches = 0, g_graphs = 0;
size_t g_bytes = 0, g_peak = 0;
bool g_capturing = false;
std::map<const void*, std::string> g_names;
std::map<std::pair<int, const void*>, int> g_limit;  // dynamic shared memory
std::map<char*, size_t> g_live;
std::vector<std::pair<std::string, int>> g_watch;
std::vector<Config> g_config;
cudaError_t g_last = cudaSuccess;

cudaError_t note(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}

bool live(const void* p) {
  auto it = g_live.upper_bound((char*)p);
  return it != g_live.begin() && (--it, (const char*)p < it->first + it->second);
}

// what lamp_create reads back of its inputs: marginals that sum to one, a largest cost of one
void create_stats(double* out) {
  for (int b = 0; b < 128; ++b) {
    double* v = out + 12 * b;
    for (int q = 0; q < 12; ++q) v[q] = b ? 0.0 : 1.0;
    v[1] = v[7] = 1.0;
    v[2] = v[8] = 0.0;
  }
}

cudaError_t launch(const void* f, size_t smem, void** args) {
  const auto lim = g_limit.find({g_device, f});
  if (smem > (size_t)(lim == g_limit.end() ? 48 * 1024 : lim->second)) return note(cudaErrorInvalidValue);
  const std::string& name = g_names[f];
  if (!g_capturing) ++g_launches;
  for (const auto& w : g_watch)
    if (name.find(w.first) != std::string::npos && !live(*(void**)args[w.second])) ++g_bad;
  if (name.find("k_create_stats") != std::string::npos) create_stats(*(double**)args[9]);
  return cudaSuccess;
}

CUresult encode_tiled(...) { return CUDA_SUCCESS; }

}  // namespace

extern "C" {

void fake_reset() {
  g_device = g_fail_attr = 0;
  g_fail_alloc = g_byte_limit = -1;
  g_bad = g_reads = g_launches = g_graph_launches = g_graphs = 0;
  g_peak = g_bytes;
  g_limit.clear();
  g_watch.clear();
}
void fake_set_device(int d) { g_device = d; }
void fake_fail_alloc(long long after) { g_fail_alloc = after; }
void fake_limit(long long bytes) { g_byte_limit = bytes; }
void fake_fail_attr(int on) { g_fail_attr = on; }
void fake_watch(const char* name, int arg) { g_watch.emplace_back(name, arg); }
long long fake_bad() { return g_bad; }
long long fake_launches() { return g_launches; }
long long fake_graph_launches() { return g_graph_launches; }
long long fake_graphs() { return g_graphs; }
// copies from device to host memory
long long fake_reads() { return g_reads; }
long long fake_bytes() { return (long long)g_bytes; }
long long fake_peak() { return (long long)g_peak; }

// ---- registration and launches ----
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, void*, void*, void*, void*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t st) {
  g_config.push_back({grid, block, smem, st});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* st) {
  const Config c = g_config.back();
  g_config.pop_back();
  *grid = c.grid;
  *block = c.block;
  *smem = c.smem;
  *(cudaStream_t*)st = c.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void** args, size_t smem, cudaStream_t) {
  return launch((const void*)k, smem, args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  return launch(f, c->dynamicSmemBytes, args);
}

// ---- device, attributes ----
cudaError_t cudaGetDevice(int* d) { return *d = g_device, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (g_fail_attr) return note(cudaErrorInvalidValue);
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) g_limit[{g_device, f}] = v;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) { return std::memset(a, 0, sizeof(*a)), cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 2, cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = (void*)encode_tiled;
  if (q) *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return *p = nullptr, cudaErrorInvalidSymbol; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "fake error"; }

// ---- memory ----
cudaError_t cudaMalloc(void** p, size_t bytes) {
  if (g_fail_alloc >= 0 && g_fail_alloc-- == 0) return note(cudaErrorMemoryAllocation);
  if (g_byte_limit >= 0 && g_bytes + bytes > (size_t)g_byte_limit) return note(cudaErrorMemoryAllocation);
  *p = std::calloc(1, bytes);
  g_live[(char*)*p] = bytes;
  g_bytes += bytes;
  if (g_bytes > g_peak) g_peak = g_bytes;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  const auto it = g_live.find((char*)p);
  if (it == g_live.end()) return ++g_bad, note(cudaErrorInvalidValue);
  g_bytes -= it->second;
  g_live.erase(it);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t bytes, unsigned) { return *p = std::calloc(1, bytes), cudaSuccess; }
cudaError_t cudaMallocHost(void** p, size_t bytes) { return *p = std::calloc(1, bytes), cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { return std::free(p), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  g_reads += kind == cudaMemcpyDeviceToHost;
  return std::memcpy(d, s, n), cudaSuccess;
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
  for (size_t i = 0; i < h; ++i) std::memcpy((char*)d + i * dp, (const char*)s + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return std::memset(p, v, n), cudaSuccess; }

// ---- streams, events, graphs ----
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return *s = (cudaStream_t)std::malloc(1), cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) { return *e = (cudaEvent_t)std::malloc(1), cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return g_capturing = true, cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  g_capturing = false;
  return *g = (cudaGraph_t)std::malloc(1), cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return std::free(g), cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  ++g_graphs;
  return *e = (cudaGraphExec_t)std::malloc(1), cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return ++g_graph_launches, cudaSuccess; }

}  // extern "C"
