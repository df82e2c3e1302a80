// A CUDA runtime without a GPU, for tests of the library's host code on the CPU: the
// library's object files are linked against this file instead of cudart.  Device memory
// is a number (allocations are counted against a limit, never touched), streams, events
// and graphs are empty, a kernel launch is recorded and does nothing.  Copies to the host
// deliver bytes 0xff (NaN, -1).
//
// As on a device, a launch with more than 48 KB of dynamic shared memory is refused
// unless cudaFuncSetAttribute has raised the kernel's limit on the current device.
#include <cuda_runtime_api.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <string>
#include <utility>
#include <vector>

namespace {

struct Launch {
  std::string name;
  unsigned grid[3];
  size_t smem;
  cudaStream_t stream;
  std::vector<int> head;   // first ints of the first argument (task-graph kernels)
};
struct State {
  int device = 0;
  size_t limit = ~(size_t)0, live = 0, peak = 0, next = (size_t)1 << 40;
  cudaError_t last = cudaSuccess;
  std::map<size_t, size_t> blocks;
  std::map<const void*, std::string> names;
  std::map<std::pair<const void*, int>, int> smem;
  std::vector<Launch> launches;
  dim3 grid, block;
  size_t shared = 0;
  cudaStream_t stream = nullptr;
};
State& st() {
  static State* s = new State;   // outlives every static destructor
  return *s;
}

cudaError_t fail(cudaError_t e) { return st().last = e; }

cudaError_t alloc(void** p, size_t bytes) {
  State& s = st();
  if (s.live + bytes > s.limit) return fail(cudaErrorMemoryAllocation);
  *p = reinterpret_cast<void*>(s.next);
  s.blocks[s.next] = bytes;
  s.next += (bytes + 511) / 512 * 512 + 512;
  s.live += bytes;
  if (s.live > s.peak) s.peak = s.live;
  return cudaSuccess;
}
cudaError_t release(void* p) {
  State& s = st();
  auto it = s.blocks.find(reinterpret_cast<size_t>(p));
  if (p && it == s.blocks.end()) return fail(cudaErrorInvalidValue);
  if (p) {
    s.live -= it->second;
    s.blocks.erase(it);
  }
  return cudaSuccess;
}

cudaError_t launch(const void* f, dim3 g, size_t smem, void** args, cudaStream_t stream) {
  State& s = st();
  if (!g.x || !g.y || !g.z || g.y > 65535 || g.z > 65535)
    return fail(cudaErrorInvalidConfiguration);
  if (smem > 48 * 1024) {
    auto it = s.smem.find({f, s.device});
    if (it == s.smem.end() || (size_t)it->second < smem) return fail(cudaErrorInvalidValue);
  }
  Launch l{s.names[f], {g.x, g.y, g.z}, smem, stream, {}};
  if (l.name.find("potrf_dag_kernel") != std::string::npos)
    l.head.assign(static_cast<int*>(args[0]), static_cast<int*>(args[0]) + 16);
  s.launches.push_back(l);
  return cudaSuccess;
}

int encode(...) { return 0; }

}  // namespace

extern "C" {

// ---- what the tests read and set -------------------------------------------
void fake_reset(size_t limit) {
  State& s = st();
  s.limit = limit;
  s.peak = s.live;
  s.last = cudaSuccess;
  s.launches.clear();
}
void fake_set_device(int d) { st().device = d; }
size_t fake_live() { return st().live; }
size_t fake_peak() { return st().peak; }
int fake_launches() { return (int)st().launches.size(); }
const char* fake_launch_name(int i) { return st().launches[i].name.c_str(); }
unsigned fake_launch_grid(int i, int d) { return st().launches[i].grid[d]; }
size_t fake_launch_stream(int i) { return reinterpret_cast<size_t>(st().launches[i].stream); }
int fake_launch_head(int i, int k) { return st().launches[i].head[k]; }

// ---- registration and launches ---------------------------------------------
void** __cudaRegisterFatBinary(void*) {
  static void* h = nullptr;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*,
                            dim3*, dim3*, int*) {
  st().names[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s) {
  st().grid = g;
  st().block = b;
  st().shared = smem;
  st().stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = st().grid;
  *b = st().block;
  *smem = st().shared;
  *static_cast<cudaStream_t*>(s) = st().stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3, void** args, size_t smem,
                               cudaStream_t s) {
  return launch(reinterpret_cast<const void*>(k), g, smem, args, s);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  return launch(f, c->gridDim, c->dynamicSmemBytes, args, c->stream);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) {
    if (v > 227 * 1024) return fail(cudaErrorInvalidValue);
    st().smem[{f, st().device}] = v;
  }
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t*) {
  *n = 76;
  return cudaSuccess;
}

// ---- device, errors ----------------------------------------------------------
cudaError_t cudaGetDevice(int* d) {
  *d = st().device;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetStreamPriorityRange(int* least, int* greatest) {
  *least = 0;
  *greatest = -5;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "error of the test runtime"; }
cudaError_t cudaGetLastError() {
  const cudaError_t e = st().last;
  st().last = cudaSuccess;
  return e;
}
cudaError_t cudaPeekAtLastError() { return st().last; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = reinterpret_cast<void*>((size_t)1 << 32);
  return cudaSuccess;
}

// ---- memory -------------------------------------------------------------------
cudaError_t cudaMalloc(void** p, size_t n) { return alloc(p, n); }
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return alloc(p, n); }
cudaError_t cudaFree(void* p) { return release(p); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return release(p); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = std::calloc(1, n);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void* p) {
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* dst, const void*, size_t n, cudaMemcpyKind k) {
  if (k == cudaMemcpyDeviceToHost) std::memset(dst, 0xff, n);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind k, cudaStream_t) {
  return cudaMemcpy(dst, src, n, k);
}
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }

// ---- streams, events, graphs -------------------------------------------------
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  static size_t n = 0;
  *s = reinterpret_cast<cudaStream_t>(++n);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* c) {
  *c = cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) { return cudaSuccess; }
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  *g = reinterpret_cast<cudaGraph_t>(1);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(1);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(1);
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 1.0f;
  return cudaSuccess;
}

}  // extern "C"
