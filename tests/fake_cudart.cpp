// A stand-in for the CUDA runtime, preloaded into a process without a GPU: device
// memory is host memory, launches run nothing but are recorded with their launch
// shape and arguments, and graphs are the launches captured into them.  It shows
// what the library's host code asks of CUDA.
#include <cuda_runtime.h>
#include <sys/mman.h>

#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <utility>
#include <vector>

namespace {

struct Launch {
  dim3 grid, block;
  size_t smem;
  void* ptr[3];  // the first three arguments, if they are pointers (batch_step_kernel)
};
struct Graph {
  std::vector<Launch> nodes;
};

std::map<char*, size_t> live;           // allocations
std::set<Graph*> graphs;                // cudaGraph_t not yet destroyed
bool capturing = false, pointers = false;
Graph* captured = nullptr;
long long fail_in = -1;                 // launches until one is refused
int device = 0;
cudaError_t last_error = cudaSuccess;
std::set<std::pair<const void*, int>> big_smem;  // kernels allowed > 48 KB, by device
std::vector<long long> last;            // shape of the last launch
int second[4];                          // and the first four words of its second argument
struct Counts {
  long long launches, stale, refused, no_attr, replayed;
} n;

bool is_live(void* p) {
  auto it = live.upper_bound(static_cast<char*>(p));
  return it != live.begin() && static_cast<char*>(p) < (--it)->first + it->second;
}

cudaError_t error(cudaError_t e) { return last_error = e; }

cudaError_t launch(const void* f, dim3 grid, dim3 block, void** args, size_t smem, bool ex) {
  if (fail_in >= 0 && fail_in-- == 0) return error(cudaErrorLaunchFailure);
  if (!grid.x || !grid.y || !grid.z || grid.x > 0x7fffffffu || grid.y > 65535 ||
      grid.z > 65535 || !block.x || block.x * block.y * block.z > 1024) {
    ++n.refused;
    return error(cudaErrorInvalidConfiguration);
  }
  if (smem > 49152 && !big_smem.count({f, device})) {
    ++n.no_attr;
    return error(cudaErrorInvalidValue);
  }
  ++n.launches;
  Launch l{grid, block, smem, {nullptr, nullptr, nullptr}};
  if (ex && pointers)
    for (int i = 0; i < 3; ++i) l.ptr[i] = *static_cast<void**>(args[i]);
  if (ex) std::memcpy(second, args[1], sizeof(second));
  last = {grid.x, grid.y, grid.z, block.x, (long long)smem};
  if (capturing) captured->nodes.push_back(l);
  return cudaSuccess;
}

}  // namespace

extern "C" {

// ---- what the tests ask ---------------------------------------------------------
void fake_pointers(int on) { pointers = on != 0; }
void fake_fail_in(long long k) { fail_in = k; }
void fake_device(int d) { device = d; }
void fake_counts(long long* out) { std::memcpy(out, &n, sizeof(n)); }
void fake_second(int* out) { std::memcpy(out, second, sizeof(second)); }
long long fake_graphs() { return (long long)graphs.size(); }
void fake_last(long long* out) { for (size_t i = 0; i < last.size(); ++i) out[i] = last[i]; }

// ---- the runtime ------------------------------------------------------------------
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
cudaError_t cudaDeviceSynchronize() { return cudaSuccess; }
cudaError_t cudaGetLastError() { return std::exchange(last_error, cudaSuccess); }
const char* cudaGetErrorString(cudaError_t) { return "refused by the stand-in"; }

cudaError_t cudaMalloc(void** p, size_t bytes) {
  // zero pages, backed when touched; never given back, so that no address returns
  void* a = mmap(nullptr, bytes ? bytes : 1, PROT_READ | PROT_WRITE,
                 MAP_PRIVATE | MAP_ANONYMOUS | MAP_NORESERVE, -1, 0);
  if (a == MAP_FAILED) return cudaErrorMemoryAllocation;
  live[static_cast<char*>(a)] = bytes ? bytes : 1;
  *p = a;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) { live.erase(static_cast<char*>(p)); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* s, size_t b, cudaMemcpyKind) {
  std::memcpy(d, s, b);
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t b, cudaMemcpyKind, cudaStream_t) {
  std::memcpy(d, s, b);
  return cudaSuccess;
}
cudaError_t cudaMemset(void*, int, size_t) { return cudaSuccess; }
cudaError_t cudaMemsetAsync(void*, int, size_t, cudaStream_t) { return cudaSuccess; }

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = reinterpret_cast<cudaStream_t>(std::malloc(1));
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) { std::free(s); return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t, cudaStreamCaptureStatus* s) {
  *s = capturing ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = reinterpret_cast<cudaEvent_t>(std::malloc(1));
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free(e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) { *ms = 1; return cudaSuccess; }

cudaError_t cudaStreamBeginCapture(cudaStream_t, cudaStreamCaptureMode) {
  captured = new Graph();
  capturing = true;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* g) {
  capturing = false;
  graphs.insert(captured);
  *g = reinterpret_cast<cudaGraph_t>(captured);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  graphs.erase(reinterpret_cast<Graph*>(g));
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t g, unsigned long long) {
  *e = reinterpret_cast<cudaGraphExec_t>(new Graph(*reinterpret_cast<Graph*>(g)));
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t e) {
  delete reinterpret_cast<Graph*>(e);
  return cudaSuccess;
}
cudaError_t cudaGraphUpload(cudaGraphExec_t, cudaStream_t) { return cudaSuccess; }
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t) {
  for (const Launch& l : reinterpret_cast<Graph*>(e)->nodes) {
    ++n.replayed;
    for (void* p : l.ptr)
      if (p && !is_live(p)) ++n.stale;
  }
  return cudaSuccess;
}

cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int) {
  big_smem.insert({f, device});
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  std::memset(a, 0, sizeof(*a));
  a->numRegs = 128;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* k, const void* f, int,
                                                                   size_t smem, unsigned) {
  *k = smem > 49152 && !big_smem.count({f, device}) ? 0 : 4;
  return cudaSuccess;
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void** args) {
  return launch(f, c->gridDim, c->blockDim, args, c->dynamicSmemBytes, true);
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = reinterpret_cast<cudaKernel_t>(const_cast<void*>(f));
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3 block, void** args, size_t smem,
                               cudaStream_t) {
  return launch(k, grid, block, args, smem, false);
}

static int fake_encode(...) { return 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** p, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* q) {
  *p = reinterpret_cast<void*>(&fake_encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

}  // extern "C"
