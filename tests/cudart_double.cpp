// The CUDA runtime calls that the library makes, answered on the host: device
// memory is host memory, kernels and copies do nothing, streams and events are
// tokens.  Linked with the library's own objects in place of libcudart, it runs
// the library's host code (plans, scratch, graphs) without a GPU, and keeps
// account of what that code allocates, frees, captures and launches.
#include <cuda_runtime_api.h>
#include <driver_types.h>

#include <cstdint>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>

namespace {

std::map<char*, size_t> live;  // device blocks
size_t limit = SIZE_MAX;       // a larger device block is refused
bool own_capture = false;      // between cudaStreamBeginCapture and EndCapture
bool user_capture = false;     // the caller's stream captures
int64_t mallocs = 0, frees = 0, instantiated = 0, graph_launches = 0, stale_launches = 0, strided = 0;

struct Graph {
  std::set<char*> blocks;  // the blocks that were live when it was captured
  bool stale = false;      // one of them has been freed since
};
std::set<Graph*> execs;

cudaError_t token(void** p) {
  *p = std::malloc(1);
  return cudaSuccess;
}

}  // namespace

extern "C" {

// ------------------------------------------------------------ for the tests
void double_limit(uint64_t bytes) { limit = bytes; }
void double_user_capture(int on) { user_capture = on != 0; }
// 0 allocations, 1 frees, 2 graphs instantiated, 3 graph launches, 4 launches of a
// graph one of whose blocks was freed after its capture, 5 copies row by row (3-D)
int64_t double_count(int k) {
  const int64_t v[] = {mallocs, frees, instantiated, graph_launches, stale_launches, strided};
  return v[k];
}

// ------------------------------------------------------------ memory
cudaError_t cudaMalloc(void** p, size_t n) {
  if (user_capture) return cudaErrorStreamCaptureUnsupported;
  if (n > limit) return cudaErrorMemoryAllocation;
  *p = std::calloc(1, 1);  // never read or written through
  live[(char*)*p] = n;
  ++mallocs;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {
  if (!p) return cudaSuccess;
  if (!live.erase((char*)p)) return cudaErrorInvalidValue;
  for (Graph* g : execs) g->stale = g->stale || g->blocks.count((char*)p) != 0;
  std::free(p);
  ++frees;
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void*) { return cudaSuccess; }
// The words that the library itself reads back (counters) are zero; arrays are not written.
cudaError_t cudaMemcpy(void* d, const void*, size_t n, cudaMemcpyKind kind) {
  if (kind == cudaMemcpyDeviceToHost && n <= 8) std::memset(d, 0, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind kind, cudaStream_t) {
  return cudaMemcpy(d, s, n, kind);
}
cudaError_t cudaMemcpy2DAsync(void*, size_t dp, const void*, size_t sp, size_t w, size_t, cudaMemcpyKind, cudaStream_t) {
  return w <= dp && w <= sp && dp <= 0x7fffffff && sp <= 0x7fffffff ? cudaSuccess : cudaErrorInvalidPitchValue;
}
cudaError_t cudaMemcpy3DAsync(const cudaMemcpy3DParms*, cudaStream_t) {
  ++strided;
  return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return token(p); }

// ------------------------------------------------------------ device
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { return *v = 152, cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof *p);
  std::strcpy(p->name, "double");
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaSuccess ? "no error" : "error of the double"; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *p = nullptr;
  if (q) *q = cudaDriverEntryPointSymbolNotFound;
  return cudaErrorSymbolNotFound;
}

// ------------------------------------------------------------ kernels
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  return *n = 2, cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void*) { return *k = nullptr, cudaSuccess; }
unsigned __cudaPushCallConfiguration(dim3, dim3, size_t, struct CUstream_st*) { return 0; }
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* stream) {
  *g = dim3(), *b = dim3(), *smem = 0, *(void**)stream = nullptr;
  return cudaSuccess;
}
void** __cudaRegisterFatBinary(void*) {
  static void* handle = nullptr;
  return &handle;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, void*, void*, void*, void*, int*) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}

// ------------------------------------------------------------ streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return token((void**)s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = own_capture || user_capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return token((void**)e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return token((void**)e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { return *ms = 1.f, cudaSuccess; }
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return own_capture = true, cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  own_capture = false;
  return token((void**)g);
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return std::free(g), cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  Graph* g = new Graph;
  for (const auto& b : live) g->blocks.insert(b.first);
  execs.insert(g);
  ++instantiated;
  *e = (cudaGraphExec_t)g;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
  execs.erase((Graph*)e);
  delete (Graph*)e;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  ++graph_launches;
  stale_launches += ((Graph*)e)->stale;
  return cudaSuccess;
}

}  // extern "C"
