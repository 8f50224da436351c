// A CUDA runtime without a device, for tests of the library's host side: the
// library's objects are linked with it instead of libcudart. Memory is host
// memory, kernels do nothing, and everything put on a stream is executed in
// order at the next synchronisation, as late as a device may. It records what
// the tests ask about (counts) and what no caller may do (violations).
#pragma once
#include <cuda_runtime_api.h>

#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <set>
#include <string>
#include <vector>

namespace fake {

enum Kind { kNone, kKernel, kCopy, kSet, kWait };
struct Op {
  Kind kind = kNone;
  void* dst = nullptr;
  const void* src = nullptr;
  size_t bytes = 0;
  int value = 0;
  bool pinned = false;         // a copy that reads page-locked memory when it runs
  std::vector<char> contents;  // what a copy is meant to read
};
struct Graph {
  std::vector<Op> ops;
};
struct Stream {
  Graph* capture = nullptr;
  Kind last = kNone;  // what was put on it last
};
struct Event {
  Graph* capture = nullptr;
};

inline std::vector<Op> queue;                  // not yet executed, in order
inline std::map<char*, size_t> pinned;         // page-locked allocations
inline std::map<const void*, std::string> names;
inline std::set<std::pair<int, const void*>> large_smem;  // (device, kernel): opted in to more than 48 KB
inline std::map<std::string, int> count;       // captures, instantiations, host allocations, kernel launches by name
inline std::vector<std::string> violations;
inline std::map<int, int> occupancy = {{0, 4}, {1, 3}};
inline Stream legacy;
inline thread_local int device = 0;
inline thread_local cudaError_t last_error = cudaSuccess;
inline bool no_pinned = false, no_graphs = false;  // no memory for them

inline void violate(const std::string& s) { violations.push_back(s); }
inline Stream* of(cudaStream_t s) { return s ? reinterpret_cast<Stream*>(s) : &legacy; }

inline void execute(const Op& o) {
  if (o.kind == kSet) std::memset(o.dst, o.value, o.bytes);
  if (o.kind != kCopy) return;
  if (o.pinned && std::memcmp(o.src, o.contents.data(), o.bytes) != 0)
    violate("page-locked memory changed before the copy that reads it ran");
  std::memmove(o.dst, o.pinned ? o.src : o.contents.data(), o.bytes);
}
inline void drain() {
  for (const Op& o : queue) execute(o);
  queue.clear();
}
inline bool is_pinned(const void* p) {
  const auto it = pinned.upper_bound((char*)p);
  if (it == pinned.begin()) return false;
  const auto q = std::prev(it);
  return (char*)p < q->first + q->second;
}
inline cudaError_t put(cudaStream_t s, Op o) {
  Stream* st = of(s);
  st->last = o.kind;
  if (st->capture) {
    st->capture->ops.push_back(std::move(o));
    return cudaSuccess;
  }
  if (o.kind == kCopy) {
    o.pinned = is_pinned(o.src);
    // the source is read now (pageable memory is staged, device memory follows in order: run what is in front)
    if (!o.pinned && !queue.empty()) drain();
    o.contents.assign((const char*)o.src, (const char*)o.src + o.bytes);
  }
  queue.push_back(std::move(o));
  return cudaSuccess;
}
inline cudaError_t launch(const void* f, dim3 grid, size_t smem, cudaStream_t s, bool early) {
  count["kernel " + names[f]]++;
  count["grid " + names[f]] = (int)grid.x;
  if (smem > 48 * 1024 && !large_smem.count({device, f})) return last_error = cudaErrorInvalidValue;
  if (early && of(s)->last != kKernel) violate(names[f] + " may start early but no kernel is in front of it");
  Op o;
  o.kind = kKernel;
  return put(s, o);
}

}  // namespace fake

extern "C" {

static dim3 fake_cfg_grid, fake_cfg_block;
static size_t fake_cfg_smem;
static cudaStream_t fake_cfg_stream;

void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char* f, char*, const char* name, int, uint3*, uint3*, dim3*, dim3*, int*) {
  std::string s = name;  // mangled: the identifier is enough
  for (const char* k : {"k_project", "k_scan_tiles", "k_refine_update", "k_pnp_scan", "k_pmm_sums", "k_composite",
                        "k_vis_backward"})
    if (s.find(k) != std::string::npos) s = k;
  fake::names[f] = s;
}
void __cudaRegisterVar(void**, char*, char*, const char*, int, size_t, int, int) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t smem, struct CUstream_st* s) {
  fake_cfg_grid = g;
  fake_cfg_block = b;
  fake_cfg_smem = smem;
  fake_cfg_stream = s;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* smem, void* s) {
  *g = fake_cfg_grid;
  *b = fake_cfg_block;
  *smem = fake_cfg_smem;
  *(cudaStream_t*)s = fake_cfg_stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) {
  *k = (cudaKernel_t)f;
  return cudaSuccess;
}
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3 grid, dim3, void**, size_t smem, cudaStream_t s) {
  return fake::launch((const void*)k, grid, smem, s, false);
}
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) {
  bool early = false;
  for (unsigned i = 0; i < c->numAttrs; ++i)
    early = early || (c->attrs[i].id == cudaLaunchAttributeProgrammaticStreamSerialization &&
                      c->attrs[i].val.programmaticStreamSerializationAllowed);
  return fake::launch(f, c->gridDim, c->dynamicSmemBytes, c->stream, early);
}
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int) {
  fake::large_smem.insert({fake::device, f});
  fake::count["cudaFuncSetAttribute"]++;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = fake::occupancy[fake::device];
  return cudaSuccess;
}

cudaError_t cudaGetDevice(int* d) {
  *d = fake::device;
  return cudaSuccess;
}
cudaError_t cudaSetDevice(int d) {
  fake::device = d;
  return cudaSuccess;
}
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) {
  *v = 152;
  return cudaSuccess;
}
cudaError_t cudaGetDeviceProperties(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  std::strcpy(p->name, "fake");
  p->multiProcessorCount = 152;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() {
  const cudaError_t e = fake::last_error;
  fake::last_error = cudaSuccess;
  return e;
}
const char* cudaGetErrorString(cudaError_t e) {
  static thread_local char s[32];
  std::snprintf(s, sizeof(s), "error %d", (int)e);
  return s;
}
cudaError_t cudaDeviceSynchronize() {
  fake::drain();
  return cudaSuccess;
}

cudaError_t cudaMalloc(void** p, size_t n) {
  fake::count["cudaMalloc"]++;
  *p = std::calloc(1, n);
  return *p ? cudaSuccess : cudaErrorMemoryAllocation;
}
cudaError_t cudaFree(void* p) {  // waits for the device
  fake::drain();
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaMallocAsync(void** p, size_t n, cudaStream_t) { return cudaMalloc(p, n); }
cudaError_t cudaFreeAsync(void* p, cudaStream_t) { return cudaFree(p); }
cudaError_t cudaHostAlloc(void** p, size_t n, unsigned) {
  fake::count["cudaMallocHost"]++;
  if (fake::no_pinned) return fake::last_error = cudaErrorMemoryAllocation;
  *p = std::calloc(1, n);
  fake::pinned[(char*)*p] = n;
  return cudaSuccess;
}
cudaError_t cudaMallocHost(void** p, size_t n) { return cudaHostAlloc(p, n, 0); }
cudaError_t cudaFreeHost(void* p) {  // not documented to wait
  const size_t n = fake::pinned[(char*)p];
  for (const fake::Op& o : fake::queue)
    if (o.pinned && (const char*)o.src >= (char*)p && (const char*)o.src < (char*)p + n) {
      fake::violate("page-locked memory freed before the copy that reads it ran");
      fake::drain();
      break;
    }
  fake::pinned.erase((char*)p);
  std::free(p);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  std::memset(a, 0, sizeof(*a));
  a->type = fake::is_pinned(p) ? cudaMemoryTypeHost : cudaMemoryTypeUnregistered;
  a->devicePointer = fake::is_pinned(p) ? (void*)p : nullptr;
  return cudaSuccess;
}
cudaError_t cudaGetSymbolAddress(void**, const void*) { return cudaErrorInvalidSymbol; }

cudaError_t cudaMemcpyAsync(void* d, const void* s, size_t n, cudaMemcpyKind, cudaStream_t st) {
  fake::Op o;
  o.kind = fake::kCopy;
  o.dst = d;
  o.src = s;
  o.bytes = n;
  return fake::put(st, o);
}
cudaError_t cudaMemcpy2DAsync(void* d, size_t dp, const void* s, size_t sp, size_t w, size_t h, cudaMemcpyKind k,
                              cudaStream_t st) {
  for (size_t i = 0; i < h; ++i) cudaMemcpyAsync((char*)d + i * dp, (const char*)s + i * sp, w, k, st);
  return cudaSuccess;
}
cudaError_t cudaMemcpy(void* d, const void* s, size_t n, cudaMemcpyKind) {
  fake::drain();
  std::memmove(d, s, n);
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* d, int v, size_t n, cudaStream_t st) {
  fake::count["cudaMemsetAsync"]++;
  fake::Op o;
  o.kind = fake::kSet;
  o.dst = d;
  o.value = v;
  o.bytes = n;
  return fake::put(st, o);
}
cudaError_t cudaMemset(void* d, int v, size_t n) {
  fake::drain();
  std::memset(d, v, n);
  return cudaSuccess;
}

cudaError_t cudaStreamCreateWithFlags(cudaStream_t* s, unsigned) {
  *s = (cudaStream_t) new fake::Stream();
  return cudaSuccess;
}
cudaError_t cudaStreamDestroy(cudaStream_t s) {
  fake::drain();
  delete fake::of(s);
  return cudaSuccess;
}
cudaError_t cudaStreamSynchronize(cudaStream_t) {
  fake::drain();
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned) {
  fake::Event* ev = (fake::Event*)e;
  fake::of(s)->capture = ev->capture;  // joins (or leaves) the capture the event belongs to
  fake::of(s)->last = fake::kWait;
  return cudaSuccess;
}
cudaError_t cudaStreamIsCapturing(cudaStream_t s, cudaStreamCaptureStatus* c) {
  *c = fake::of(s)->capture ? cudaStreamCaptureStatusActive : cudaStreamCaptureStatusNone;
  return cudaSuccess;
}
cudaError_t cudaEventCreate(cudaEvent_t* e) {
  *e = (cudaEvent_t) new fake::Event();
  return cudaSuccess;
}
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { return cudaEventCreate(e); }
cudaError_t cudaEventDestroy(cudaEvent_t e) {
  delete (fake::Event*)e;
  return cudaSuccess;
}
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  ((fake::Event*)e)->capture = fake::of(s)->capture;
  return cudaSuccess;
}
cudaError_t cudaEventSynchronize(cudaEvent_t) {
  fake::drain();
  return cudaSuccess;
}
cudaError_t cudaEventElapsedTime(float* ms, cudaEvent_t, cudaEvent_t) {
  *ms = 0.001f;
  return cudaSuccess;
}

cudaError_t cudaStreamBeginCapture(cudaStream_t s, cudaStreamCaptureMode) {
  fake::count["captures"]++;
  fake::of(s)->capture = new fake::Graph();
  fake::of(s)->last = fake::kNone;
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t s, cudaGraph_t* g) {
  *g = (cudaGraph_t)fake::of(s)->capture;
  fake::of(s)->capture = nullptr;
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* x, cudaGraph_t g, unsigned long long) {
  if (fake::no_graphs) return fake::last_error = cudaErrorMemoryAllocation;
  *x = (cudaGraphExec_t) new fake::Graph(*(fake::Graph*)g);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t x, cudaStream_t s) {
  fake::count["replays"]++;
  for (const fake::Op& o : ((fake::Graph*)x)->ops) fake::put(s, o);
  return cudaSuccess;
}
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }  // kept: streams forked in a capture may name it
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t x) {
  delete (fake::Graph*)x;
  return cudaSuccess;
}

static int fake_encode() { return 0; }
cudaError_t cudaGetDriverEntryPointByVersion(const char*, void** f, unsigned, unsigned long long,
                                             cudaDriverEntryPointQueryResult* r) {
  *f = (void*)fake_encode;
  *r = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}

}  // extern "C"
