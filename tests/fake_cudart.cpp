// A CUDA runtime for host tests of the library's memory handling: device
// memory is host memory with a settable capacity, copies are memcpy, kernels
// do not run but their names and grids are recorded.  Linked with the
// library's objects in the place of the CUDA runtime (test_memory_limits.py).
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
std::map<void*, size_t> g_live;
size_t g_used = 0, g_peak = 0, g_capacity = ~(size_t)0;
long long g_allocs = 0, g_fail_at = -1;   // the allocation (counted from 0) that fails
std::vector<std::string> g_launched;
std::string g_text;
cudaError_t g_last = cudaSuccess;
bool g_no_cooperative = false;
dim3 g_grid, g_block;
size_t g_smem;
cudaStream_t g_stream;

// (filled by the objects' own initialisers, in any order)
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
template <class T>
T handle() {
  return reinterpret_cast<T>(std::malloc(1));
}
cudaError_t set(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}
cudaError_t launch(const void* f, dim3 grid, dim3 block) {
  if (!grid.x || !grid.y || !grid.z || !block.x) return set(cudaErrorInvalidConfiguration);
  auto it = names().find(f);
  g_launched.push_back(it == names().end() ? "?" : it->second);
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- the test's side ----
void fake_set_capacity(size_t n) { g_capacity = n; }
void fake_fail_at(long long k) { g_fail_at = k < 0 ? -1 : g_allocs + k; }
void fake_no_cooperative(int on) { g_no_cooperative = on != 0; }
size_t fake_used(void) { return g_used; }
size_t fake_peak(void) { return g_peak; }
void fake_reset_peak(void) { g_peak = g_used; }
// launched kernels since the last call, one mangled name per line
const char* fake_launched(void) {
  g_text.clear();
  for (auto& s : g_launched) g_text += s + "\n";
  g_launched.clear();
  return g_text.c_str();
}

// ---- memory ----
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_allocs++ == g_fail_at || n > g_capacity || g_used > g_capacity - n) return set(cudaErrorMemoryAllocation);
  *p = std::calloc(n ? n : 1, 1);
  if (!*p) std::abort();   // (the host, not the test's capacity)
  g_live[*p] = n;
  g_used += n;
  if (g_used > g_peak) g_peak = g_used;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  auto it = g_live.find(p);
  if (it == g_live.end()) std::abort();   // freed twice, or never allocated
  g_used -= it->second;
  g_live.erase(it);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) {
  *p = std::calloc(n, 1);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  if (!d || !s) return set(cudaErrorInvalidValue);
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  if (!p) return set(cudaErrorInvalidValue);
  std::memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = nullptr;
  return set(cudaErrorInvalidSymbol);
}

// ---- streams, events, graphs ----
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = handle<cudaStream_t>();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  std::free(s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = handle<cudaEvent_t>();
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  std::free(e);
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.0f;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) {
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  if (g) *g = handle<cudaGraph_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) {
  *g = handle<cudaGraph_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  std::free(g);
  return cudaSuccess;
}
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t* n) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = handle<cudaGraphExec_t>();
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
  std::free(e);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  g_launched.push_back("graph");
  return cudaSuccess;
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
  *h = 0;
  return cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams*) {
  return set(cudaErrorNotSupported);
}

// ---- device ----
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152
       : a == cudaDevAttrCooperativeLaunch ? 1
       : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448
                                                      : 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError(void) {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "error of the test runtime"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = nullptr;
  if (q) *q = cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}

// ---- kernels ----
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeCooperative && g_no_cooperative)
      return set(cudaErrorCooperativeLaunchTooLarge);
  return launch(f, c->gridDim, c->blockDim);
}
cudaError_t cudaLaunchKernel(const void* f, dim3 grid, dim3 block, void**, size_t, cudaStream_t) {
  return launch(f, grid, block);
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void**, size_t, cudaStream_t) {
  return launch((const void*)k, grid, block);
}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, struct CUstream_st* s) {
  g_grid = grid;
  g_block = block;
  g_smem = smem;
  g_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  *grid = g_grid;
  *block = g_block;
  *smem = g_smem;
  *(cudaStream_t*)s = g_stream;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names()[f] = name;
}
}
