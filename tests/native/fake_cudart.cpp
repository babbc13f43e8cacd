// A stand-in for the CUDA runtime that the library is linked against in tests of its host code
// (test_host_faults.py): no GPU, kernels and copies do nothing, every stream and event is always
// finished.  It keeps the runtime's last error as the real one does (set by a failing call, cleared
// by cudaGetLastError alone), logs calls and kernel launches, and fails a call on request.
#include <cuda.h>
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {

struct Launch {
  std::string name;
  unsigned grid;
  bool overlap;
  void* stream;
  void* second;  // the second pointer of the argument block: the destination of a copy kernel
};
struct Range {
  size_t bytes;
  cudaMemoryType type;
};

std::map<std::string, int> g_count, g_fail_at, g_fail_with;
std::map<const void*, std::string> g_names, g_loaded;
std::map<const char*, Range> g_mem;
std::vector<Launch> g_log;
cudaError_t g_last = cudaSuccess;
void* g_capturing = nullptr;
struct {
  dim3 grid, block;
  size_t smem;
  void* stream;
} g_config;

cudaError_t done(cudaError_t e) {
  if (e != cudaSuccess) g_last = e;
  return e;
}

cudaError_t step(const char* name) {
  const int k = g_count[name]++;
  const auto it = g_fail_at.find(name);
  if (it == g_fail_at.end() || it->second != k) return cudaSuccess;
  g_fail_at.erase(it);
  return done(static_cast<cudaError_t>(g_fail_with[name]));
}

template <typename T>
cudaError_t handle(const char* name, T* out) {
  const cudaError_t e = step(name);
  if (e == cudaSuccess) *out = reinterpret_cast<T>(std::malloc(16));
  return e;
}

cudaError_t alloc(const char* name, void** out, size_t bytes, cudaMemoryType type) {
  const cudaError_t e = step(name);
  if (e != cudaSuccess) return e;
  *out = std::calloc(1, bytes + 256);
  g_mem[static_cast<const char*>(*out)] = Range{bytes, type};
  return cudaSuccess;
}

cudaMemoryType type_of(const void* p) {
  auto it = g_mem.upper_bound(static_cast<const char*>(p));
  if (it == g_mem.begin()) return cudaMemoryTypeUnregistered;
  --it;
  return static_cast<const char*>(p) < it->first + it->second.bytes ? it->second.type : cudaMemoryTypeUnregistered;
}

void load(const void* fn) { g_loaded[fn] = g_names[fn]; }

cudaError_t launch(const char* call, const void* fn, unsigned grid, bool overlap, void* stream, void** args) {
  const cudaError_t e = step(call);
  if (e != cudaSuccess) return e;
  load(fn);
  void* second = nullptr;
  if (g_names[fn].find("k_sm_copy") != std::string::npos) second = static_cast<void**>(args[0])[1];
  g_log.push_back(Launch{g_names[fn], grid, overlap, stream, second});
  return cudaSuccess;
}

CUresult fake_cuLaunchKernelEx(const CUlaunchConfig* c, CUfunction f, void** args, void**) {
  const cudaError_t e = launch("cuLaunchKernelEx", f, c->gridDimX, c->numAttrs > 0, c->hStream, args);
  return e == cudaSuccess ? CUDA_SUCCESS : CUDA_ERROR_UNKNOWN;
}

CUresult fake_cuPointerGetAttributes(unsigned n, CUpointer_attribute* what, void** into, CUdeviceptr p) {
  g_count["cuPointerGetAttributes"]++;
  const cudaMemoryType t = type_of(reinterpret_cast<const void*>(p));
  for (unsigned i = 0; i < n; ++i)
    if (what[i] == CU_POINTER_ATTRIBUTE_MEMORY_TYPE)
      *static_cast<CUmemorytype*>(into[i]) = t == cudaMemoryTypeDevice ? CU_MEMORYTYPE_DEVICE
                                             : t == cudaMemoryTypeHost ? CU_MEMORYTYPE_HOST
                                                                       : static_cast<CUmemorytype>(0);
  return CUDA_SUCCESS;
}

}  // namespace

extern "C" {

// ---- the test's side -------------------------------------------------------------------
// Call number `after` from now (0: the next one) of `name` fails with `err`.
void fake_fail(const char* name, int after, int err) {
  g_fail_at[name] = g_count[name] + after;
  g_fail_with[name] = err;
}
int fake_count(const char* name) { return g_count[name]; }
void fake_leave_error(int err) { g_last = static_cast<cudaError_t>(err); }
void fake_capturing(void* stream) { g_capturing = stream; }
int fake_launches(const char* part, unsigned* grid, int* overlap) {
  int n = 0;
  for (const Launch& l : g_log)
    if (l.name.find(part) != std::string::npos) {
      ++n;
      if (grid) *grid = l.grid;
      if (overlap) *overlap = l.overlap;
    }
  return n;
}
// Destination of the last copy kernel.
void* fake_copied_to() {
  void* p = nullptr;
  for (const Launch& l : g_log)
    if (l.second) p = l.second;
  return p;
}
int fake_loaded(const char* part) {
  int n = 0;
  for (const auto& l : g_loaded) n += l.second.find(part) != std::string::npos;
  return n;
}

// ---- registration and launches ---------------------------------------------------------
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t stream) {
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
cudaError_t __cudaGetKernel(cudaKernel_t* out, const void* fn) {
  *out = reinterpret_cast<cudaKernel_t>(const_cast<void*>(fn));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t fn, dim3 grid, dim3, void** args, size_t, cudaStream_t s) {
  return launch("launch", fn, grid.x, false, s, args);
}
cudaError_t cudaLaunchKernel(const void* fn, dim3 grid, dim3, void** args, size_t, cudaStream_t s) {
  return launch("launch", fn, grid.x, false, s, args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** args) {
  return launch("launch", fn, c->gridDim.x, c->numAttrs > 0, c->stream, args);
}
cudaError_t cudaGetFuncBySymbol(cudaFunction_t* out, const void* fn) {
  const cudaError_t e = step("cudaGetFuncBySymbol");
  if (e != cudaSuccess) return e;
  load(fn);
  *out = reinterpret_cast<cudaFunction_t>(const_cast<void*>(fn));
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void* fn) {
  const cudaError_t e = step("cudaFuncGetAttributes");
  if (e != cudaSuccess) return e;
  load(fn);
  *a = cudaFuncAttributes{};
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return step("cudaFuncSetAttribute"); }
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  static char symbol[64 * 1024];
  *p = symbol;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char* name, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *r = cudaDriverEntryPointSuccess;
  *f = !std::strcmp(name, "cuLaunchKernelEx") ? reinterpret_cast<void*>(&fake_cuLaunchKernelEx)
                                              : reinterpret_cast<void*>(&fake_cuPointerGetAttributes);
  return cudaSuccess;
}

// ---- device, memory ----------------------------------------------------------------------
cudaError_t cudaGetLastError() {
  const cudaError_t e = g_last;
  g_last = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t) { return "error of the stand-in runtime"; }
cudaError_t cudaGetDeviceCount(int* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof *p);
  std::strcpy(p->name, "none");
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrAsyncEngineCount ? 3 : 1;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return step("cudaDeviceSynchronize"); }
cudaError_t cudaMalloc(void** p, size_t n) { return alloc("cudaMalloc", p, n, cudaMemoryTypeDevice); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return alloc("cudaHostAlloc", p, n, cudaMemoryTypeHost); }
cudaError_t cudaFree(void* p) {
  g_mem.erase(static_cast<const char*>(p));
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaFreeHost(void* p) {
  g_count["cudaFreeHost"]++;
  return cudaFree(p);
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) { return *d = h, cudaSuccess; }
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::memset(a, 0, sizeof *a);
  a->type = type_of(p);
  return cudaSuccess;
}
cudaError_t cudaMemset(void* p, int v, size_t n) { return std::memset(p, v, n), cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) { return std::memcpy(d, s, n), cudaSuccess; }
cudaError_t cudaMemcpyAsync(void*, const void*, size_t, cudaMemcpyKind, cudaStream_t) { return step("cudaMemcpyAsync"); }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return step("cudaMemsetAsync"); }
cudaError_t cudaLaunchHostFunc(cudaStream_t, cudaHostFn_t, void*) { return step("cudaLaunchHostFunc"); }

// ---- streams, events ---------------------------------------------------------------------
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle("cudaStreamCreateWithFlags", s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t s) {
  const cudaError_t e = step("cudaStreamSynchronize");
  return s && s == g_capturing ? done(cudaErrorStreamCaptureUnsupported) : e;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return step("cudaStreamWaitEvent"); }
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* st) {
  *st = s && s == g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return step("cudaStreamIsCapturing");
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t s, cudaStreamCaptureStatus* st, unsigned long long*, cudaGraph_t*,
                                     const cudaGraphNode_t**, const cudaGraphEdgeData**, size_t*) {
  return cudaStreamIsCapturing(s, st);
}
cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle("cudaEventCreate", e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle("cudaEventCreate", e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return step("cudaEventRecord"); }
cudaError_t cudaEventQuery(cudaEvent_t) { return step("cudaEventQuery"); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return step("cudaEventSynchronize"); }
// every measurement is shorter than the one before it
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  const cudaError_t e = step("cudaEventElapsedTime");
  *ms = 1.0f / (float)g_count["cudaEventElapsedTime"];
  return e;
}

// ---- graphs ------------------------------------------------------------------------------
cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { return handle("cudaGraphCreate", g); }
cudaError_t cudaGraphDestroy(cudaGraph_t g) { return std::free(g), cudaSuccess; }
cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t,
                                   const cudaKernelNodeParams* p) {
  load(p->func);
  return handle("cudaGraphAddKernelNode", n);
}
cudaError_t cudaGraphAddMemcpyNode1D(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, void*, const void*,
                                     size_t, cudaMemcpyKind) {
  return handle("cudaGraphAddMemcpyNode1D", n);
}
cudaError_t cudaGraphAddMemsetNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, const cudaMemsetParams*) {
  return handle("cudaGraphAddMemsetNode", n);
}
cudaError_t cudaGraphAddHostNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, size_t, const cudaHostNodeParams*) {
  return handle("cudaGraphAddHostNode", n);
}
cudaError_t cudaGraphGetNodes(cudaGraph_t, cudaGraphNode_t*, size_t* n) { return *n = 1, cudaSuccess; }
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  return handle("cudaGraphInstantiate", e);
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaGraphExecUpdate(cudaGraphExec_t, cudaGraph_t, cudaGraphExecUpdateResultInfo*) {
  return step("cudaGraphExecUpdate");
}
cudaError_t cudaGraphExecMemcpyNodeSetParams1D(cudaGraphExec_t, cudaGraphNode_t, void*, const void*, size_t, cudaMemcpyKind) {
  return step("cudaGraphExecMemcpyNodeSetParams1D");
}
cudaError_t cudaGraphNodeSetEnabled(cudaGraphExec_t, cudaGraphNode_t, unsigned) { return step("cudaGraphNodeSetEnabled"); }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t s) {
  const cudaError_t e = step("cudaGraphLaunch");
  return s && s == g_capturing ? done(cudaErrorStreamCaptureUnsupported) : e;
}

}  // extern "C"
