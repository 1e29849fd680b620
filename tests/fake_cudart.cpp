// A CUDA runtime on host memory, for tests of the library's host code without a GPU: linked with the
// library's own objects in place of the CUDA runtime (see fake_runtime.py).
//
// "Device" memory is host memory.  Asynchronous copies and clears run as late as the runtime's contract
// allows: at the next synchronising call, in issue order, reading their source then.  Kernels do
// nothing but leave a record of their launch.  A launched graph finishes what it would work on: every
// batch slot at the start of a step is done, every solve state ends with the status the test asked for.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdlib>
#include <cstring>
#include <functional>
#include <map>
#include <mutex>
#include <string>
#include <vector>

#include "rd_internal.h"
#include "rd_launch.h"

namespace {

std::recursive_mutex g_mu;
std::map<char*, size_t> g_allocs;
std::vector<std::function<void()>> g_pending;
std::map<const void*, std::string> g_names;    // host stub -> mangled kernel name
std::vector<std::string> g_launched;           // names of the launched kernels, in order
std::vector<std::string> g_attr;               // kernels whose shared-memory limit was raised
std::map<std::string, float> g_cost;           // part of a kernel's name -> time of a launch
std::map<void*, size_t> g_events;              // event -> launches when it was recorded
bool g_refuse_alloc = false;
bool g_hold = false;                           // graphs leave the slots as they are
long g_alloc_calls = 0;                        // cudaMalloc and cudaFree
size_t g_slots = 0;                            // slots of the batch under test
int g_state_status[2] = {rd::ST_CONVERGED, rd::ST_CONVERGED};
thread_local int g_capturing = 0;

using Lock = std::lock_guard<std::recursive_mutex>;

void run_pending() {
  Lock lk(g_mu);
  std::vector<std::function<void()>> ops;
  ops.swap(g_pending);
  for (auto& f : ops) f();
}

void finish_graph() {
  Lock lk(g_mu);
  for (auto& [p, n] : g_allocs) {
    if (g_slots && !g_hold && n == g_slots * sizeof(rd::Slot)) {
      for (size_t k = 0; k < g_slots; ++k) {
        rd::Slot& s = reinterpret_cast<rd::Slot*>(p)[k];
        if (s.phase != rd::PH_BEGIN) continue;
        s.phase = rd::PH_DONE;
        s.steps_done = s.nsteps;
      }
    }
    if (n == 3 * sizeof(rd::State))
      for (int k = 0; k < 2; ++k) reinterpret_cast<rd::State*>(p)[k].status = g_state_status[k];
  }
}

cudaError_t allocate(void** p, size_t n) {
  Lock lk(g_mu);
  *p = nullptr;
  if (posix_memalign(p, 4096, n ? n : 1)) return cudaErrorMemoryAllocation;
  if (n < (1u << 26)) std::memset(*p, 0, n);
  g_allocs[static_cast<char*>(*p)] = n;
  return cudaSuccess;
}

void enqueue(std::function<void()> f) {
  if (g_capturing) return;  // a graph's copies and clears: part of what finish_graph stands for
  Lock lk(g_mu);
  g_pending.push_back(std::move(f));
}

void launched(const void* fn) {
  Lock lk(g_mu);
  g_launched.push_back(g_names[fn]);
}

template <class H>
cudaError_t handle(H* h) {
  *h = reinterpret_cast<H>(std::malloc(16));
  return cudaSuccess;
}

CUresult encode_stub(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                     const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                     CUtensorMapFloatOOBfill) {
  return CUDA_SUCCESS;
}

struct Config {
  dim3 grid, block;
  size_t smem;
  cudaStream_t stream;
};
thread_local std::vector<Config> g_configs;
void* g_fatbin;
char g_symbol[4 << 20];

}  // namespace

extern "C" {

// --- what the tests set and read ---
void fake_refuse_alloc(int on) { g_refuse_alloc = on; }
void fake_hold(int on) {
  Lock lk(g_mu);
  g_hold = on;
}
long fake_alloc_calls() { return g_alloc_calls; }
void fake_slots(size_t n) { g_slots = n; }
void fake_status(int outer, int inner) { g_state_status[0] = outer, g_state_status[1] = inner; }
void fake_cost(const char* part, float t) { g_cost[part] = t; }
// the names recorded, one per line
static size_t names_out(const std::vector<std::string>& v, char* out, size_t cap) {
  std::string s;
  for (const std::string& n : v) s += n + "\n";
  if (out && cap) std::strncpy(out, s.c_str(), cap - 1);
  return s.size() + 1;
}
size_t fake_launched(char* out, size_t cap) { return names_out(g_launched, out, cap); }
size_t fake_limits(char* out, size_t cap) { return names_out(g_attr, out, cap); }
// whether some device allocation holds these bytes
int fake_contains(const void* bytes, size_t n) {
  Lock lk(g_mu);
  for (auto& [p, len] : g_allocs)
    if (memmem(p, len, bytes, n)) return 1;
  return 0;
}
int fake_outer_after_inner(int inner) { return rd::outer_after_inner(inner); }
// The plan of k_primal for bands of `rows` rows: whether it runs, and its shared memory.
int fake_plan_band(int elem, int nx, int ny, int nc, int H, int rows, int limit, int* smem_primal) {
  rd::Desc d{};
  d.nx = nx, d.ny = ny, d.ncomp = nc;
  while ((1 << d.lognx) < nx) ++d.lognx;
  while ((1 << d.logny) < ny) ++d.logny;
  d.col_width = 2;
  d.band_rows = d.upd_rows = rows;
  rd::LaunchCfg c{};
  c.transform = 1;
  if (elem == 4) rd::plan_band<float>(d, H, limit, c);
  else rd::plan_band<double>(d, H, limit, c);
  *smem_primal = c.smem_primal;
  return c.fast_row;
}

// --- the runtime ---
void** __cudaRegisterFatBinary(void*) { return &g_fatbin; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  Lock lk(g_mu);
  g_names[host] = name;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 grid, dim3 block, size_t smem, cudaStream_t s) {
  g_configs.push_back({grid, block, smem, s});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* grid, dim3* block, size_t* smem, void* s) {
  const Config c = g_configs.back();
  g_configs.pop_back();
  *grid = c.grid, *block = c.block, *smem = c.smem;
  *static_cast<cudaStream_t*>(s) = c.stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* fn) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(fn));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t, cudaStream_t) {
  launched(reinterpret_cast<const void*>(k));
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void* fn, void**) {
  launched(fn);
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  std::memset(a, 0, sizeof(*a));
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void* fn, cudaFuncAttribute, int) {
  Lock lk(g_mu);
  g_attr.push_back(g_names[fn]);
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { return *d = 0, cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : a == cudaDevAttrMultiProcessorCount ? 152 : 1;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t e) { return e == cudaErrorMemoryAllocation ? "out of memory" : "error"; }
cudaError_t cudaGetSymbolAddress(void** p, const void*) { return *p = g_symbol, cudaSuccess; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** fn, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *fn = reinterpret_cast<void*>(&encode_stub);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t n) {
  ++g_alloc_calls;
  return g_refuse_alloc ? cudaErrorMemoryAllocation : allocate(p, n);
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) { return allocate(p, n + 16); }
static cudaError_t release(void* p) {
  run_pending();
  Lock lk(g_mu);
  g_allocs.erase(static_cast<char*>(p));
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { return ++g_alloc_calls, release(p); }
cudaError_t cudaFreeHost(void* p) { return release(p); }
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  run_pending();
  std::memcpy(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t) {
  enqueue([=] { std::memcpy(d, s, n); });
  return cudaSuccess;
}
cudaError_t cudaMemset(void* d, int v, size_t n) { return run_pending(), std::memset(d, v, n), cudaSuccess; }
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t) {
  enqueue([=] { std::memset(d, v, n); });
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return run_pending(), cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) { return handle(s); }
cudaError_t cudaStreamDestroy(cudaStream_t s) { return std::free(s), cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return run_pending(), cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* st) {
  *st = g_capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return ++g_capturing, cudaSuccess; }
cudaError_t cudaStreamBeginCaptureToGraph(cudaStream_t, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                                          cudaStreamCaptureMode) {
  return ++g_capturing, cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) { return --g_capturing, handle(g); }
cudaError_t cudaStreamGetCaptureInfo(cudaStream_t, cudaStreamCaptureStatus* st, unsigned long long*, cudaGraph_t*,
                                     const cudaGraphNode_t**, const cudaGraphEdgeData**, size_t*) {
  *st = cudaStreamCaptureStatusActive;
  return cudaSuccess;
}
cudaError_t cudaStreamUpdateCaptureDependencies(cudaStream_t, cudaGraphNode_t*, const cudaGraphEdgeData*, size_t, unsigned) {
  return cudaSuccess;
}

cudaError_t cudaEventCreate(cudaEvent_t* e) { return handle(e); }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return handle(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { return std::free(e), cudaSuccess; }
cudaError_t cudaEventRecordWithFlags(cudaEvent_t e, cudaStream_t, unsigned) {
  Lock lk(g_mu);
  g_events[e] = g_launched.size();
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) { return cudaEventRecordWithFlags(e, s, 0); }
// the launches between the two events, each at the cost the test gave its kernel (1 without)
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  Lock lk(g_mu);
  *ms = 0.f;
  for (size_t k = g_events[a]; k < g_events[b]; ++k) {
    float t = 1.f;
    for (auto& [part, cost] : g_cost)
      if (g_launched[k].find(part) != std::string::npos) t = cost;
    *ms += t;
  }
  return cudaSuccess;
}

cudaError_t cudaGraphCreate(cudaGraph_t* g, unsigned) { return handle(g); }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphConditionalHandleCreate(cudaGraphConditionalHandle* h, cudaGraph_t, unsigned, unsigned) {
  return *h = 1, cudaSuccess;
}
cudaError_t cudaGraphAddNode(cudaGraphNode_t* n, cudaGraph_t, const cudaGraphNode_t*, const cudaGraphEdgeData*, size_t,
                             cudaGraphNodeParams* p) {
  static cudaGraph_t body[1];
  if (p->type == cudaGraphNodeTypeConditional) p->conditional.phGraph_out = body;
  return handle(n);
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t, unsigned long long) { return handle(x); }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) { return std::free(x), cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) {
  enqueue(finish_graph);
  return cudaSuccess;
}

}  // extern "C"
