// A CUDA runtime of the host's own for tests of the library's host code: streams, events, copies, launches and graphs
// are written down in a log instead of being run (device memory is host memory, copies are made), any call can be made
// to fail, and so can any allocation.  The kernel sources are not part of this library: their launch builders are
// stand-ins that note what the launch would compute.
#include <cuda.h>
#include <cuda_runtime.h>

#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <new>
#include <string>
#include <vector>

#include "kernels.h"

namespace {
struct Event { int id; };
struct Stream { int id; };
struct Node { size_t at; struct Graph* of; char what[256]; };
struct Graph { std::vector<Node*> nodes; };
struct State {
  std::string log, replayed;  // replayed: the launches of the graphs, one by one
  std::map<std::string, long> fail_in;  // function -> calls until one fails
  long alloc_in = -1;
  int events = 0, streams = 100;
  cudaStream_t capturing = nullptr;
  Graph* graph = nullptr;
  long encodes = 0;
  int sms = 148, pairs = 74;
  size_t pageable_from = 0, pageable_to = 0;
};
State* g = nullptr;  // (never freed: the library may be used until the process ends)
State& s() {
  if (!g) g = new (std::malloc(sizeof(State))) State();
  return *g;
}
void note(const char* fmt, ...) {
  char b[512];
  va_list a;
  va_start(a, fmt);
  std::vsnprintf(b, sizeof(b), fmt, a);
  va_end(a);
  const long keep = s().alloc_in;
  s().alloc_in = -1;  // the log's own memory is not part of the test
  s().log += b;
  s().log += '\n';
  s().alloc_in = keep;
}
bool fails(const char* fn) {
  const long keep = s().alloc_in;
  s().alloc_in = -1;
  auto it = s().fail_in.find(fn);
  const bool now = it != s().fail_in.end() && --it->second == 0;
  s().alloc_in = keep;
  return now;
}
template <class T, class... A>
T* plain_new(A... a) { return new (std::malloc(sizeof(T))) T{a...}; }
#define FAILS(fn) if (fails(#fn)) return cudaErrorUnknown

CUresult encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  ++s().encodes;
  return CUDA_SUCCESS;
}
long sid(cudaStream_t st) { return (long)(intptr_t)st; }
const char kKernels[8] = {};  // addresses that stand for kernels
}  // namespace

// the library's own allocations (it is linked so that its calls come here)
static void* allocate(size_t n, size_t align) {
  if (g && g->alloc_in > 0 && --g->alloc_in == 0) throw std::bad_alloc();
  void* p = std::aligned_alloc(align, (n + align) / align * align);
  if (!p) throw std::bad_alloc();
  return p;
}
void* operator new(size_t n) { return allocate(n, 16); }
void* operator new(size_t n, std::align_val_t a) { return allocate(n, (size_t)a); }
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, size_t) noexcept { std::free(p); }
void operator delete(void* p, std::align_val_t) noexcept { std::free(p); }
void operator delete(void* p, size_t, std::align_val_t) noexcept { std::free(p); }

extern "C" {
const char* fake_log() { return s().log.c_str(); }
const char* fake_replayed() { return s().replayed.c_str(); }
void fake_reset() { s().log.clear(); s().replayed.clear(); s().fail_in.clear(); s().alloc_in = -1; s().encodes = 0; s().pageable_from = s().pageable_to = 0; }
void fake_fail(const char* fn, long nth) { s().fail_in[fn] = nth; }
void fake_fail_alloc(long nth) { s().alloc_in = nth; }
long fake_alloc_left() { return s().alloc_in; }
void fake_sms(int n) { s().sms = n; }  // before the library has looked at the device
void fake_pageable(size_t from, size_t to) { s().pageable_from = from, s().pageable_to = to; }  // other host memory is pinned
void fake_pairs(int n) { s().pairs = n; }  // CTA pairs that the device holds at once
long fake_encodes() { return s().encodes; }

cudaError_t cudaGetDeviceCount(int* n) { *n = 1; return cudaSuccess; }
cudaError_t cudaSetDevice(int) { return cudaSuccess; }
cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
cudaError_t cudaGetDeviceProperties_v2(cudaDeviceProp* p, int) {
  std::memset(p, 0, sizeof(*p));
  p->major = 10;
  p->multiProcessorCount = s().sms;
  return cudaSuccess;
}
cudaError_t cudaGetDriverEntryPoint(const char*, void** fn, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *fn = (void*)encode;
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
const char* cudaGetErrorString(cudaError_t) { return "made to fail"; }
cudaError_t cudaDeviceGetStreamPriorityRange(int* l, int* h) { *l = 0; *h = -1; return cudaSuccess; }
cudaError_t cudaStreamCreateWithFlags(cudaStream_t* st, unsigned) { *st = (cudaStream_t)(intptr_t)++s().streams; return cudaSuccess; }
cudaError_t cudaStreamCreateWithPriority(cudaStream_t* st, unsigned, int) { *st = (cudaStream_t)(intptr_t)++s().streams; return cudaSuccess; }
cudaError_t cudaStreamDestroy(cudaStream_t) { return cudaSuccess; }
cudaError_t cudaStreamSynchronize(cudaStream_t st) { note("sync %ld", sid(st)); return cudaSuccess; }
cudaError_t cudaEventCreateWithFlags(cudaEvent_t* e, unsigned) { *e = (cudaEvent_t)plain_new<Event>(++s().events); return cudaSuccess; }
cudaError_t cudaEventDestroy(cudaEvent_t e) { std::free((void*)e); return cudaSuccess; }
cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t st) {
  FAILS(cudaEventRecord);
  note("record %d %ld", ((Event*)e)->id, sid(st));
  return cudaSuccess;
}
cudaError_t cudaStreamWaitEvent(cudaStream_t st, cudaEvent_t e, unsigned) {
  FAILS(cudaStreamWaitEvent);
  note("wait %d %ld", ((Event*)e)->id, sid(st));
  return cudaSuccess;
}
cudaError_t cudaMemsetAsync(void* p, int v, size_t n, cudaStream_t) { std::memset(p, v, n); return cudaSuccess; }
cudaError_t cudaMemcpy(void* d, const void* src, size_t n, cudaMemcpyKind) { std::memcpy(d, src, n); return cudaSuccess; }
cudaError_t cudaMemcpyAsync(void* d, const void* src, size_t n, cudaMemcpyKind k, cudaStream_t st) {
  FAILS(cudaMemcpyAsync);
  std::memmove(d, src, n);
  note("%s %ld %zu %zu %zu", k == cudaMemcpyHostToDevice ? "h2d" : "d2h", sid(st), (size_t)d, (size_t)src, n);
  return cudaSuccess;
}
cudaError_t cudaPointerGetAttributes(cudaPointerAttributes* a, const void* p) {
  FAILS(cudaPointerGetAttributes);
  a->type = (size_t)p >= s().pageable_from && (size_t)p < s().pageable_to ? cudaMemoryTypeUnregistered : cudaMemoryTypeHost;
  return cudaSuccess;
}
cudaError_t cudaGetLastError() { return cudaSuccess; }
cudaError_t cudaGetSymbolAddress(void** p, const void* sym) { *p = const_cast<void*>(sym); return cudaSuccess; }

cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void*, void** args) {
  FAILS(cudaLaunchKernelExC);
  if (s().capturing && c->stream == s().capturing) {
    const long keep = s().alloc_in;
    s().alloc_in = -1;
    Node* nd = plain_new<Node>(s().graph->nodes.size(), s().graph);
    std::snprintf(nd->what, sizeof(nd->what), "%s", (const char*)args[0]);
    s().graph->nodes.push_back(nd);
    s().alloc_in = keep;
  } else {
    note("launch %ld %s", sid(c->stream), (const char*)args[0]);
  }
  return cudaSuccess;
}
cudaError_t cudaStreamBeginCapture(cudaStream_t st, cudaStreamCaptureMode) {
  FAILS(cudaStreamBeginCapture);
  s().capturing = st;
  s().graph = plain_new<Graph>();
  return cudaSuccess;
}
cudaError_t cudaStreamEndCapture(cudaStream_t, cudaGraph_t* out) {
  s().capturing = nullptr;
  *out = (cudaGraph_t)s().graph;
  return cudaSuccess;
}
cudaError_t cudaGraphGetNodes(cudaGraph_t gr, cudaGraphNode_t*, size_t* n) { *n = ((Graph*)gr)->nodes.size(); return cudaSuccess; }
cudaError_t cudaGraphGetRootNodes(cudaGraph_t gr, cudaGraphNode_t* out, size_t* n) {
  *out = (cudaGraphNode_t)((Graph*)gr)->nodes.at(0);
  *n = 1;
  return cudaSuccess;
}
cudaError_t cudaGraphNodeGetDependentNodes_v2(cudaGraphNode_t nd, cudaGraphNode_t* out, cudaGraphEdgeData*, size_t* n) {
  Node* x = (Node*)nd;
  const bool last = x->at + 1 == x->of->nodes.size();
  *n = last ? 0 : 1;
  if (out && !last) *out = (cudaGraphNode_t)x->of->nodes[x->at + 1];
  return cudaSuccess;
}
cudaError_t cudaGraphInstantiate(cudaGraphExec_t* e, cudaGraph_t gr, unsigned long long) {
  FAILS(cudaGraphInstantiate);
  *e = (cudaGraphExec_t)gr;
  return cudaSuccess;
}
cudaError_t cudaGraphExecKernelNodeSetParams(cudaGraphExec_t, cudaGraphNode_t nd, const cudaKernelNodeParams* p) {
  std::snprintf(((Node*)nd)->what, sizeof(Node::what), "%s", (const char*)p->kernelParams[0]);
  return cudaSuccess;
}
cudaError_t cudaGraphLaunch(cudaGraphExec_t e, cudaStream_t st) {
  FAILS(cudaGraphLaunch);
  note("launch %ld graph %zu", sid(st), ((Graph*)e)->nodes.size());
  const long keep = s().alloc_in;
  s().alloc_in = -1;
  s().replayed += "graph\n";
  for (const Node* nd : ((Graph*)e)->nodes) s().replayed += std::string("launch - ") + nd->what + '\n';
  s().alloc_in = keep;
  return cudaSuccess;
}
cudaError_t cudaGraphExecDestroy(cudaGraphExec_t) { return cudaSuccess; }
cudaError_t cudaGraphDestroy(cudaGraph_t) { return cudaSuccess; }
}

namespace qe {
namespace {
Launch named(const char* fmt, ...) {
  char b[256] = {};
  va_list a;
  va_start(a, fmt);
  std::vsnprintf(b, sizeof(b), fmt, a);
  va_end(a);
  Launch l;
  l.func = kKernels;
  l.params.resize(sizeof(b));
  std::memcpy(l.params.data(), b, sizeof(b));
  l.nbytes = sizeof(b);
  return l;
}
}  // namespace
bool whole_row_tiles(uint32_t M) { return M % 256 == 0; }
cudaError_t gemm_prepare() { return cudaSuccess; }
bool chained_fit(int sms, cudaStream_t) { return s().pairs >= sms / 2; }
uint32_t gemm_width(const GemmDesc*, uint32_t, int) { return 1; }
Launch make_quantize(const QuantParams&) { return named("cast 1"); }
Launch make_quantize_multi(const QuantParams*, uint32_t n, const Announce& early) {
  return early.word ? named("cast %u early %u", n, early.count) : named("cast %u", n);
}
// (a GEMM launch is "gemm <problems> products <products>", and then what it does with the count of commits)
uint32_t announce_commits(Launch* l, uint32_t*) {
  std::strcat((char*)l->params.data(), " announces");
  return (uint32_t)std::atoi((char*)l->params.data() + 5);
}
void withdraw_commits(Launch* l, uint32_t*) { std::strcat((char*)l->params.data(), " withdraws"); }
Launch make_commit(const CommitParams&) { return named("commit"); }
Launch make_status_gather(const StatusGatherParams&) { return named("status"); }
Launch make_amax_pass1(const AmaxParams&) { return named("amax1"); }
Launch make_amax_pass2(const AmaxParams&) { return named("amax2"); }
Launch make_accumulate(const AccumParams&) { return named("accumulate"); }
Launch make_arena_reduce(const ArenaReduceParams&) { return named("arena"); }
Launch make_gemm(const GemmDesc& d, int) { return named("gemm 1 products %u", d.nseg); }
bool make_gemm_group(const GemmDesc* p, uint32_t n, int, Launch* out) {
  uint32_t ops = 0;
  for (uint32_t i = 0; i < n; ++i) ops += p[i].nseg;
  *out = named("gemm %u products %u", n, ops);
  return true;
}
}  // namespace qe
