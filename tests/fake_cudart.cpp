// A CUDA runtime that runs nothing: the library's objects linked against it run
// their host code on a machine without a GPU.  Device memory is host memory,
// kernel launches are recorded, and a launch or a heap allocation can be made to
// fail.
#include <cuda.h>
#include <cuda_runtime_api.h>
#include <cxxabi.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <iterator>
#include <map>
#include <new>
#include <string>

namespace {
std::map<const void*, std::string>& names() {
  static std::map<const void*, std::string> m;
  return m;
}
std::string& log() {
  static std::string s;
  return s;
}
std::map<size_t, void*>& last_alloc() {
  static std::map<size_t, void*> m;
  return m;
}
int g_launches_left = -1;          // launches that still succeed; -1: all
thread_local bool g_heap_fails = false;
struct Call {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
} g_call;

cudaError_t launch(const void* f, dim3 g, dim3 b, size_t smem, int cluster, bool pdl) {
  if (g_launches_left == 0) return cudaErrorInvalidValue;
  if (g_launches_left > 0) --g_launches_left;
  const bool fails = g_heap_fails;
  g_heap_fails = false;              // (for this log's own allocations)
  const auto it = names().find(f);
  char line[512];
  snprintf(line, sizeof line, "%s|%u,%u,%u|%u|%zu|%d|%d\n", it == names().end() ? "?" : it->second.c_str(), g.x, g.y,
           g.z, b.x, smem, cluster, pdl ? 1 : 0);
  log() += line;
  g_heap_fails = fails;
  return cudaSuccess;
}
CUresult encode_tiled(...) { return CUDA_SUCCESS; }
}  // namespace

void* operator new(size_t n) {
  if (g_heap_fails) throw std::bad_alloc();
  if (void* p = malloc(n ? n : 1)) return p;
  throw std::bad_alloc();
}
void* operator new(size_t n, const std::nothrow_t&) noexcept { return g_heap_fails ? nullptr : malloc(n ? n : 1); }
void operator delete(void* p) noexcept { free(p); }
void operator delete(void* p, size_t) noexcept { free(p); }

extern "C" {
// ------------------------------------------------------------ for the tests
// the launches since the last clear: "kernel|grid x,y,z|threads|shared bytes|cluster CTAs|dependent" lines
const char* fake_launches() { return log().c_str(); }
void fake_clear() { log().clear(); }
void fake_launches_left(int n) { g_launches_left = n; }
void fake_heap_fails(int on) { g_heap_fails = on != 0; }
// the last live device allocation of that size
void* fake_last_alloc(size_t bytes) { return last_alloc().count(bytes) ? last_alloc()[bytes] : nullptr; }

// ------------------------------------------------------------ the runtime
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  int st = 0;
  char* d = abi::__cxa_demangle(name, nullptr, nullptr, &st);
  names()[host] = st == 0 ? d : name;
  free(d);
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s) {
  g_call = Call{g, b, smem, s};
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = g_call.grid;
  *b = g_call.block;
  *smem = g_call.smem;
  *static_cast<cudaStream_t*>(s) = g_call.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t) {
  return launch(reinterpret_cast<const void*>(k), g, b, smem, 1, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  int cluster = 1;
  bool pdl = false;
  for (unsigned i = 0; i < c->numAttrs; ++i) {
    const cudaLaunchAttribute& a = c->attrs[i];
    if (a.id == cudaLaunchAttributeClusterDimension)
      cluster = a.val.clusterDim.x * a.val.clusterDim.y * a.val.clusterDim.z;
    if (a.id == cudaLaunchAttributeProgrammaticStreamSerialization) pdl = a.val.programmaticStreamSerializationAllowed;
  }
  return launch(f, c->gridDim, c->blockDim, c->dynamicSmemBytes, cluster, pdl);
}
// 152 SMs; clusters of 1..8 CTAs at one CTA per SM, as a GB300 reports them
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* c) {
  static const int most[9] = {0, 152, 76, 46, 36, 28, 23, 15, 15};
  int cluster = 1;
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeClusterDimension)
      cluster = c->attrs[i].val.clusterDim.x * c->attrs[i].val.clusterDim.y * c->attrs[i].val.clusterDim.z;
  *n = cluster <= 8 ? most[cluster] : 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *f = reinterpret_cast<void*>(&encode_tiled);
  if (r) *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = aligned_alloc(256, (n + 255) / 256 * 256);
  if (!*p) return cudaErrorMemoryAllocation;
  last_alloc()[n] = *p;
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = malloc(n);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) {
  for (auto it = last_alloc().begin(); it != last_alloc().end();)
    it = it->second == p ? last_alloc().erase(it) : std::next(it);
  free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) { return cudaFree(p); }
cudaError_t cudaMemset(void* p, int v, size_t n) {
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(d, s, n, k);
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind,
                              cudaStream_t) {
  for (size_t i = 0; i < h; ++i) memcpy(static_cast<char*>(d) + i * dp, static_cast<const char*>(s) + i * sp, w);
  return cudaSuccess;
}
cudaError_t cudaMemcpyToSymbol(const void* sym, const void* s, size_t n, size_t o, cudaMemcpyKind) {
  memcpy(static_cast<char*>(const_cast<void*>(sym)) + o, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyFromSymbol(void* d, const void* sym, size_t n, size_t o, cudaMemcpyKind) {
  memcpy(d, static_cast<const char*>(sym) + o, n);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) {
  *p = const_cast<void*>(sym);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  a->type = cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaStreamCreate(cudaStream_t* s) {
  *s = nullptr;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "an error of the fake runtime"; }
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = nullptr;
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}
cudaError_t cudaEventRecordWithFlags(cudaEvent_t, cudaStream_t, unsigned) { return cudaSuccess; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
}
