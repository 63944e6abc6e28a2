// A stand-in for the CUDA runtime, on the CPU, for tests of the library's host code.
//
// The library's objects are linked against this file in place of the CUDA runtime.  Device memory is
// host memory that is never reused, so a pointer that outlived its allocation is always seen;
// kernels do not run, but every launch of a step kernel, direct or through a graph, is checked
// (its descriptors and work items must be live and their upload ordered before it) and recorded.  An
// allocation can be made to fail.  Time is a cost of the launches: every work item costs its
// threads times its planes and a start, and planes beyond a kernel's best chunk (16 node-wise,
// 32 tiled) cost more.
#include <cuda_runtime.h>
#include <string.h>

#include <cstdio>
#include <cstdlib>
#include <map>
#include <set>
#include <string>
#include <vector>

#include "../paper_1602_07483_gb300/csrc/lbpf_plan.h"

namespace {

struct Launch {
  std::string name;
  unsigned blocks = 0, threads = 0;
  cudaStream_t stream = nullptr;
  const void* ptr[3] = {};  // descriptors, work items, the one-launch ticket order
  int nptr = 0;
};
struct Record {
  std::string name;
  unsigned blocks, threads;
  int z_first, z_longest;  // planes of the first and of the longest work item
};
struct Graph {
  std::vector<Launch> launches;
};
struct Event {
  double at = 0;
};

constexpr size_t kCopied = 64u << 20;  // larger copies move nothing: no test reads them

std::map<const char*, size_t> g_live;
std::set<const void*> g_pending;  // uploads on the default stream that nothing has waited for
std::map<const void*, std::string> g_name;
std::vector<Record> g_log;
std::vector<std::string> g_bad;
std::map<cudaStream_t, Graph*> g_capture;
int g_fail_in = -1, g_fail_for = 0;  // allocations until the failing ones, and their number
double g_clock = 0;
struct Config {
  dim3 g, b;
  size_t smem;
  cudaStream_t st;
};
std::vector<Config> g_config;

size_t live_bytes(const void* p) {
  auto it = g_live.find((const char*)p);
  return it == g_live.end() ? 0 : it->second;
}

void run(const Launch& l) {
  for (int k = 0; k < l.nptr; ++k) {
    if (!live_bytes(l.ptr[k])) {
      g_bad.push_back(l.name + ": argument " + std::to_string(k) + " is not allocated");
      return;
    }
    if (g_pending.count(l.ptr[k])) g_bad.push_back(l.name + ": argument " + std::to_string(k) + " may still be uploading");
  }
  const lbpf::WorkItem* it = (const lbpf::WorkItem*)l.ptr[1];
  const bool one = l.nptr == 3;  // its grid is the resident blocks, not the items
  if (!one && live_bytes(it) < l.blocks * sizeof(*it)) {
    g_bad.push_back(l.name + ": more blocks than work items");
    return;
  }
  const bool nodes = l.name.find("_node") != std::string::npos || l.name.find("_pair") != std::string::npos ||
                     l.name.find("_moment") != std::string::npos;
  const int best = nodes ? 16 : 32;
  Record r{l.name, l.blocks, l.threads, it[0].z1 - it[0].z0, 0};
  for (unsigned k = 0; k < (one ? 1u : l.blocks); ++k) {
    const int n = it[k].z1 - it[k].z0;
    r.z_longest = n > r.z_longest ? n : r.z_longest;
    g_clock += l.threads * (n + 2.0 + 4.0 * (n > best ? n - best : 0));
  }
  g_log.push_back(r);
}

void launched(const Launch& l) {
  auto it = g_capture.find(l.stream);
  if (it != g_capture.end()) it->second->launches.push_back(l);
  else run(l);
}

// A launch of a step kernel (k_phi..., k_uth..., k_step); the others read no work items.
cudaError_t launch(const std::string& name, dim3 g, dim3 b, cudaStream_t st, void** args) {
  if (g.x == 0) return cudaErrorInvalidConfiguration;
  const bool one = name.find("k_step") != std::string::npos;
  if (!one && name.find("k_phi") == std::string::npos && name.find("k_uth") == std::string::npos) return cudaSuccess;
  Launch l;
  l.name = name;
  l.blocks = g.x;
  l.threads = b.x * b.y;
  l.stream = st;
  l.ptr[0] = *(void**)args[0];
  l.ptr[1] = *(void**)args[1];
  l.ptr[2] = one ? *(void**)args[2] : nullptr;
  l.nptr = one ? 3 : 2;
  launched(l);
  return cudaSuccess;
}

void move_bytes(void* dst, const void* src, size_t n) {
  if (n < kCopied) memcpy(dst, src, n);
}

}  // namespace

extern "C" {

// ---- the tests' side
void fake_fail_malloc(int after, int count) {  // let `after` allocations pass, then fail `count`
  g_fail_in = after;
  g_fail_for = count;
}
int fake_violations() { return (int)g_bad.size(); }
const char* fake_violation(int i) { return g_bad[i].c_str(); }
int fake_launches() { return (int)g_log.size(); }
const char* fake_launch(int i) {
  static char buf[512];
  const Record& r = g_log[i];
  snprintf(buf, sizeof buf, "%s %u %u %d %d", r.name.c_str(), r.blocks, r.threads, r.z_first, r.z_longest);
  return buf;
}
void fake_clear() {
  g_log.clear();
  g_bad.clear();
}

// ---- registration and launch stubs of compiled kernels
void** __cudaRegisterFatBinary(void*) {
  static void* h;
  return &h;
}
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
void __cudaRegisterFunction(void**, const char* host, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  g_name[host] = name;
}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* st) {
  g_config.push_back({g, b, smem, st});
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* st) {
  const Config c = g_config.back();
  g_config.pop_back();
  *g = c.g;
  *b = c.b;
  *smem = c.smem;
  *(cudaStream_t*)st = c.st;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* host) {
  *k = (cudaKernel_t)host;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 g, dim3 b, void** args, size_t, cudaStream_t st) {
  return launch(g_name[(const void*)k], g, b, st, args);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* fn, void** args) {
  return launch(g_name[fn], c->gridDim, c->blockDim, c->stream, args);
}

// ---- memory
cudaError_t cudaMalloc(void** p, size_t n) {
  if (g_fail_in == 0 && g_fail_for > 0) {
    --g_fail_for;
    *p = nullptr;
    return cudaErrorMemoryAllocation;
  }
  if (g_fail_in > 0) --g_fail_in;
  *p = calloc(n ? n : 1, 1);
  g_live[(const char*)*p] = n ? n : 1;
  return cudaSuccess;
}
cudaError_t cudaFree(void* p) {  // waits for the device
  g_pending.clear();
  g_live.erase((const char*)p);
  return cudaSuccess;
}
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  *p = calloc(n, 1);
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void* p) {
  free(p);
  return cudaSuccess;
}
cudaError_t cudaHostGetDevicePointer(void** d, void* h, unsigned) {
  *d = h;
  return cudaSuccess;
}
// on the default stream; an upload from pageable memory may return before it has arrived
cudaError_t cudaMemcpy(void* dst, const void* src, size_t n, cudaMemcpyKind kind) {
  move_bytes(dst, src, n);
  if (kind == cudaMemcpyHostToDevice) g_pending.insert(dst);
  else g_pending.clear();
  return cudaSuccess;
}
cudaError_t cudaMemcpyAsync(void* dst, const void* src, size_t n, cudaMemcpyKind, cudaStream_t) {
  move_bytes(dst, src, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) {
  if (live_bytes(p) < n) g_bad.push_back("a memset of what is not allocated");
  else if (n < kCopied) memset(p, v, n);
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void** p, const void*) {
  *p = nullptr;
  return cudaErrorInvalidSymbol;
}

// ---- device
cudaError_t cudaGetDeviceCount(int* n) {
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) {
  *d = 0;
  return cudaSuccess;
}
cudaError_t cudaDeviceSynchronize() {
  g_pending.clear();
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : a == cudaDevAttrMaxSharedMemoryPerBlockOptin ? 232448 : 0;
  return cudaSuccess;
}
cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, const void*) {
  memset(a, 0, sizeof *a);
  return cudaSuccess;
}
cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, const void*, int, size_t) {
  *n = 2;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
const char* cudaGetErrorString(cudaError_t) { return "fake error"; }

// ---- streams, events, graphs
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t)malloc(1);
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamWaitEvent(cudaStream_t, cudaEvent_t, unsigned) { return cudaSuccess; }
cudaError_t cudaStreamIsCapturing(cudaStream_t st, cudaStreamCaptureStatus* c) {
  *c = g_capture.count(st) ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t) new Event;
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  delete (Event*)e;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t) {
  ((Event*)e)->at = g_clock;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) { return cudaSuccess; }
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t a, cudaEvent_t b) {
  *ms = (float)((((Event*)b)->at - ((Event*)a)->at) * 1e-9);
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t st, cudaStreamCaptureMode) {
  g_capture[st] = new Graph;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t st, cudaGraph_t* g) {
  *g = (cudaGraph_t)g_capture[st];
  g_capture.erase(st);
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long) {
  *x = (cudaGraphExec_t) new Graph(*(Graph*)g);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t g) {
  delete (Graph*)g;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
  delete (Graph*)x;
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t) {
  for (const Launch& l : ((Graph*)x)->launches) run(l);
  return cudaSuccess;
}

}  // extern "C"
