// A CUDA runtime without a GPU for tests of the library's host code: device memory is host memory, launches are counted
// and do nothing, streams are in order at once, and a test can have a call refused. Linked with the library's own
// objects into a library of its own.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>

namespace {
std::set<void*> live;                       // device allocations
std::map<const void*, std::string> kernels;  // by host stub
std::map<std::string, long> launched;        // by (mangled) kernel name
const void* refused_dst = nullptr;           // asynchronous copies to this address are refused
bool refuse_cooperative = false, refuse_graph = false;
long syncs = 0, graph_launches = 0;
void (*on_copy)(void*, const void*, size_t) = nullptr;  // after every copy from the device

cudaError_t launch(const void* func) {
  ++launched[kernels[func]];
  return cudaSuccess;
}
CUresult encode_map(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                    const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}
cudaError_t copy(void* dst, const void* src, size_t n, cudaMemcpyKind kind) {
  memcpy(dst, src, n);
  if (kind == cudaMemcpyDeviceToHost && on_copy) on_copy(dst, src, n);
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---- what a test sets and reads ----
long fake_live() { return (long)live.size(); }
long fake_syncs() { return syncs; }
long fake_graph_launches() { return graph_launches; }
void fake_refuse_copy(const void* dst) { refused_dst = dst; }
void fake_refuse_cooperative(int on) { refuse_cooperative = on != 0; }
void fake_refuse_graph(int on) { refuse_graph = on != 0; }
void fake_on_copy(void (*f)(void*, const void*, size_t)) { on_copy = f; }
void* fake_device_buffer(size_t n) {
  void* p = nullptr;
  return cudaMalloc(&p, n) == cudaSuccess ? p : nullptr;
}
void fake_free(void* p) { cudaFree(p); }
long fake_launches(const char* part) {  // of kernels with `part` in their names
  long n = 0;
  for (auto& k : launched)
    if (k.first.find(part) != std::string::npos) n += k.second;
  return n;
}

// ---- memory ----
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = calloc(n ? n : 1, 1);
  live.insert(*p);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (p && !live.erase(p)) return cudaErrorInvalidValue;
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return (*p = calloc(n ? n : 1, 1)) ? cudaSuccess : cudaErrorMemoryAllocation; }
cudaError_t cudaFreeHost(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) {
  memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { return cudaMemset(p, v, n); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return copy(d, s, n, k); }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind k, cudaStream_t) {
  if (refused_dst && d == refused_dst) return cudaErrorInvalidValue;
  return copy(d, s, n, k);
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  memset(a, 0, sizeof *a);
  a->type = live.count(const_cast<void*>(p)) ? cudaMemoryTypeDevice : cudaMemoryTypeUnregistered;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void* symbol) {
  *p = const_cast<void*>(symbol);
  return cudaSuccess;
}

// ---- device ----
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrComputeCapabilityMajor ? 10 : a == cudaDevAttrComputeCapabilityMinor ? 3 : 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  ++syncs;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "refused"; }
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 76;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  const bool ok = !strcmp(name, "cuTensorMapEncodeTiled");
  *f = ok ? reinterpret_cast<void*>(encode_map) : nullptr;
  if (r) *r = ok ? cudaDriverEntryPointSuccess : cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}

// ---- streams, events, graphs ----
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(16);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  ++syncs;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(16);
  return cudaSuccess;
}
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.f;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = reinterpret_cast<cudaGraph_t>(16);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(16);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  if (refuse_graph) return cudaErrorCooperativeLaunchTooLarge;
  ++graph_launches;
  return cudaSuccess;
}

// ---- launches ----
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* func, void**) {
  for (unsigned i = 0; i < c->numAttrs; ++i)
    if (c->attrs[i].id == cudaLaunchAttributeCooperative && c->attrs[i].val.cooperative && refuse_cooperative)
      return cudaErrorCooperativeLaunchTooLarge;
  return launch(func);
}
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, void*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3*, dim3*, size_t*, void*) { return cudaSuccess; }
cudaError_t __cudaGetKernel(void** k, const void* func) {
  *k = const_cast<void*>(func);
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(void* k, dim3, dim3, void**, size_t, cudaStream_t) { return launch(k); }
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  kernels[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
}
