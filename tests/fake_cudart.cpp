// A stand-in for the CUDA runtime, for host tests of the library's own host code: linked with the library's
// objects in place of the real one.  Memory is host memory, kernels do nothing, streams and graphs are counted.
// Every kernel launch and memset is recorded under the kernel's name; a chosen call can be made to fail.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <vector>

namespace {
struct Launch { std::string kernel; unsigned grid, block; size_t smem; int dependent; };
struct Graph { std::vector<Launch> nodes; };
std::map<const void*, std::string> names;
std::map<std::string, size_t> opt_in;                // largest dynamic shared memory allowed
std::vector<Launch> ran;                             // what has run, graphs included
std::map<cudaStream_t, Graph*> capture;
std::map<std::string, int> calls;
std::string fail_call;
int fail_nth = 0;
cudaError_t last = cudaSuccess;
int open_captures = 0;
int null_graphs = 0;                                 // calls on no graph
std::map<cudaStream_t, bool> invalid;                // captures that another thread's call has invalidated
char pool[4096];
size_t handles = 0;

template <class T> T handle() { return (T)(pool + handles++ % sizeof pool); }

// the nth call of `what` fails
cudaError_t call(const char* what, cudaError_t e = cudaErrorInvalidValue) {
  const int n = ++calls[what];
  if (fail_call == what && n == fail_nth) { last = e; return e; }
  return cudaSuccess;
}
cudaError_t launch(const std::string& k, dim3 g, dim3 b, size_t smem, cudaStream_t st, int dep) {
  if (cudaError_t e = call(k == "memset" ? "memset" : "launch")) return e;
  const Launch l{k, g.x * g.y * g.z, b.x * b.y * b.z, smem, dep};
  auto c = capture.find(st);
  (c == capture.end() ? ran : c->second->nodes).push_back(l);
  return cudaSuccess;
}
}  // namespace

extern "C" {
// ---------------------------------------------------------------- for the test
void fake_reset() { ran.clear(); calls.clear(); fail_call.clear(); fail_nth = 0; last = cudaSuccess; null_graphs = 0; }
int fake_null_graphs() { return null_graphs; }
void fake_fail(const char* what, int nth) { calls.clear(); fail_call = what; fail_nth = nth; }
int fake_calls(const char* what) { return calls[what]; }
int fake_open_captures() { return open_captures; }
int fake_ran() { return (int)ran.size(); }
const char* fake_kernel(int i) { return ran[i].kernel.c_str(); }
long long fake_smem(int i) { return (long long)ran[i].smem; }
int fake_block(int i) { return (int)ran[i].block; }
int fake_grid(int i) { return (int)ran[i].grid; }
long long fake_opt_in(const char* kernel) { return opt_in.count(kernel) ? (long long)opt_in[kernel] : -1; }

// ---------------------------------------------------------------- kernels
void** __cudaRegisterFatBinary(void*) { return handle<void**>(); }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  names[host] = name;
}
static dim3 cfg_grid, cfg_block;
static size_t cfg_smem;
static void* cfg_stream;
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* st) {
  cfg_grid = g; cfg_block = b; cfg_smem = smem; cfg_stream = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  *g = cfg_grid; *b = cfg_block; *smem = cfg_smem; *(void**)st = cfg_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) { *k = (cudaKernel_t)host; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void**, size_t smem, cudaStream_t st) {
  return launch(names[(const void*)k], g, b, smem, st, 0);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  return launch(names[f], c->gridDim, c->blockDim, c->dynamicSmemBytes, c->stream, c->numAttrs);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) opt_in[names[f]] = (size_t)v;
  return call("cudaFuncSetAttribute");
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { const cudaError_t e = last; last = cudaSuccess; return e; }
cudaError_t cudaPeekAtLastError() { return last; }
const char* cudaGetErrorString(cudaError_t) { return "an error of the stand-in runtime"; }

// ---------------------------------------------------------------- devices and memory
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  memset(p, 0, sizeof *p);
  strcpy(p->name, "stand-in");
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *f = nullptr;
  *q = cudaDriverEntryPointSymbolNotFound;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void**, const void*) { return call("cudaGetSymbolAddress", cudaErrorInvalidSymbol); }
cudaError_t cudaMalloc(void** p, size_t n) {
  *p = aligned_alloc(256, (n + 255) / 256 * 256);
  return call("cudaMalloc", cudaErrorMemoryAllocation);
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaMalloc(p, n); }
cudaError_t cudaFree(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaFreeHost(void* p) { free(p); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  memcpy(d, s, n);
  return call("cudaMemcpyAsync");
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind k) { return cudaMemcpyAsync(d, s, n, k, nullptr); }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  if (!capture.count(st)) memset(d, v, n);
  return launch("memset", 1, 1, 0, st, 0);
}
cudaError_t cudaMemset(void* d, int v, size_t n) { memset(d, v, n); return cudaSuccess; }

// ---------------------------------------------------------------- streams and events
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = handle<cudaStream_t>();
  return call("cudaStreamCreateWithFlags");
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return call("cudaStreamSynchronize", cudaErrorLaunchFailure); }
cudaError_t cudaEventCreate(cudaEvent_t* e) { *e = handle<cudaEvent_t>(); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
// an event's time is the number of the last launch, so times compare by what ran in between (cudaEventElapsedTime)
static std::map<cudaEvent_t, size_t> event_at;
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) { event_at[e] = ran.size(); return cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t s, unsigned) { return cudaEventRecord(e, s); }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
// 1 ms a launch, 2 where a name given by fake_slow is part of the kernel's and its block is smaller than given
static std::string slow_name;
static unsigned slow_block = 0;
void fake_slow(const char* part, int block) { slow_name = part; slow_block = (unsigned)block; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = 0.f;
  for (size_t k = event_at[a]; k < event_at[b] && k < ran.size(); ++k)
    *ms += slow_block && ran[k].kernel.find(slow_name) != std::string::npos && ran[k].block < slow_block ? 2.f : 1.f;
  return cudaSuccess;
}

// ---------------------------------------------------------------- capture and graphs
cudaError_t cudaStreamBeginCapture(cudaStream_t st, cudaStreamCaptureMode) {
  if (cudaError_t e = call("cudaStreamBeginCapture")) return e;
  capture[st] = new Graph();
  ++open_captures;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t st, cudaGraph_t g, const cudaGraphNode_t*, const cudaGraphEdgeData*,
                                          size_t, cudaStreamCaptureMode) {
  if (cudaError_t e = call("cudaStreamBeginCaptureToGraph")) return e;
  capture[st] = (Graph*)g;
  ++open_captures;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t st, cudaGraph_t* g) {
  *g = nullptr;
  if (!capture.count(st)) { last = cudaErrorIllegalState; return last; }
  const bool bad = invalid[st];
  *g = bad ? nullptr : (cudaGraph_t)capture[st];
  invalid[st] = false;
  capture.erase(st);
  --open_captures;
  if (bad) return last = cudaErrorStreamCaptureInvalidated;
  return call("cudaStreamEndCapture", cudaErrorStreamCaptureInvalidated);
}
cudaError_t cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus* s) {
  *s = capture.count(st) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t st, cudaStreamCaptureStatus* s, unsigned long long*, cudaGraph_t* g,
                                     const cudaGraphNode_t** deps, const cudaGraphEdgeData** ed, size_t* n) {
  cudaStreamIsCapturing(st, s);
  if (call("invalidated") != cudaSuccess) { invalid[st] = true; last = cudaSuccess; }
  if (invalid[st]) *s = cudaStreamCaptureStatusInvalidated;
  if (g) *g = capture.count(st) && !invalid[st] ? (cudaGraph_t)capture[st] : nullptr;
  if (deps) *deps = nullptr;
  if (ed) *ed = nullptr;
  if (n) *n = 0;
  return call("cudaStreamGetCaptureInfo");
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t*, const cudaGraphEdgeData*, size_t, unsigned) {
  return call("cudaStreamUpdateCaptureDependencies");
}
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t g, unsigned, unsigned) {
  *h = ++handles;
  if (!g) ++null_graphs;
  return call("cudaGraphConditionalHandleCreate");
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t* n, cudaGraph_t g, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
  if (!g) ++null_graphs;
  *n = handle<cudaGraphNode_t>();
  cudaGraph_t* body = new cudaGraph_t((cudaGraph_t) new Graph());   // kept: a test's few
  p->conditional.phGraph_out = body;
  return call("cudaGraphAddNode");
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long) {
  *x = (cudaGraphExec_t) new Graph(*(Graph*)g);
  return call("cudaGraphInstantiate");
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
  for (const Launch& l : ((Graph*)x)->nodes) ran.push_back(l);
  return call("cudaGraphLaunch");
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) { delete (Graph*)g; return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { delete (Graph*)x; return cudaSuccess; }
}
