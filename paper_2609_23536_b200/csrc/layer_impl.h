// Internals shared by the translation units of the layer API: the context and layer objects, the launch builders of
// the three actions and the execution layer (eager launches or CUDA graphs, bracketed by the two-way stream handshake).
#pragma once
#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <vector>

#include "contract.h"
#include "error.h"
#include "kernels.h"
#include "qe.h"

using qe::fail;

#define QE_CUDA(expr)                                                                         \
  do {                                                                                        \
    cudaError_t e_ = (expr);                                                                  \
    if (e_ != cudaSuccess) return fail(QE_ERR_CUDA, "%s: %s", #expr, cudaGetErrorString(e_)); \
  } while (0)

namespace qe_impl {


typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

struct DeviceInfo {
  bool ready = false;
  int device = -1, num_sms = 0, cc_major = 0;
  EncodeTiledFn encode = nullptr;
};

int32_t device_info(int device, DeviceInfo** out);
int32_t current_device_info(DeviceInfo** d);
// Operand tensors of one shape, `apart` bytes from one to the next (one tensor: any).
struct Slots {
  const void* first;
  uint32_t count = 1;
  uint64_t apart = 0;
};
int32_t make_a_map(const DeviceInfo* d, CUtensorMap* map, const Slots& t, uint64_t M, uint64_t Kc, bool mn, uint32_t width);
int32_t make_b_map(const DeviceInfo* d, CUtensorMap* map, const Slots& t, uint64_t N, uint64_t Kc, bool mn, uint32_t width);
int32_t make_a_maps(const DeviceInfo* d, CUtensorMap* maps, const Slots& t, uint64_t M, uint64_t Kc, bool mn);
int32_t make_b_maps(const DeviceInfo* d, CUtensorMap* maps, const Slots& t, uint64_t N, uint64_t Kc, bool mn);
int32_t make_out_map(const DeviceInfo* d, CUtensorMap* map, const void* ptr, uint64_t M, uint64_t N, uint64_t ldo, bool fp32, uint32_t rows = 32);
int32_t make_out_map_u8(const DeviceInfo* d, CUtensorMap* map, const void* ptr, uint64_t M, uint64_t N, uint64_t ld);
inline uint64_t align_up(uint64_t v, uint64_t a) { return (v + a - 1) / a * a; }
inline bool shape_ok(uint32_t v) { return v >= 256 && v % 128 == 0 && v <= (1u << 20); }

}  // namespace qe_impl
using qe_impl::DeviceInfo;

// ================================================================================================ execution layer
struct ActionGraph {
  bool built = false;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
  std::vector<cudaGraphNode_t> nodes;
  std::vector<qe::Launch> launches;
};

struct qe_ctx {
  DeviceInfo* dev = nullptr;
  uint32_t exec_mode = QE_EXEC_EAGER;
  cudaStream_t exec_stream = nullptr;
  bool owns_stream = true;
  bool one_way = false;              // QE_CTX_UNSAFE_ONE_WAY_HANDOFF
  bool chained_fit = false;          // a launch of chained GEMMs can have all its blocks on the device at once
  bool launch_failed = false;        // a whole-step call's: counts of commits in device memory may not be what they should be
  uint32_t step_window = 4;          // qe_step_run: units looked ahead when planning rounds (1: action by action)
  cudaStream_t dw_stream = nullptr;  // only with QE_CTX_OVERLAP_DW
  cudaEvent_t ev_dw_in = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  // host-buffer calls: copy streams and their events, created by the first such call
  cudaStream_t h2d_stream = nullptr, d2h_stream = nullptr;
  cudaEvent_t ev_h2d = nullptr, ev_kernels = nullptr, ev_d2h = nullptr;
  bool kernels_recorded = false;
  struct HostRange { uintptr_t lo, hi; };
  std::vector<HostRange> readbacks;  // host memory that read-backs write which no upload has been ordered after yet
  qe_registry* registry = nullptr;
  qe_stats stats{};
  // Layers keep their context alive: it is released when the caller has destroyed it AND its last layer is gone,
  // so the two destroy calls may come in either order.
  uint32_t layers = 0;
  bool closed = false;
  // whole-step graphs, one per distinct (layers, actions) list
  struct StepGraph { uint64_t key; ActionGraph g; };
  std::vector<StepGraph*> step_graphs;
};

struct qe_layer {
  qe_ctx* ctx = nullptr;
  qe_layer_config cfg{};
  qe_contract* contract = nullptr;
  uint64_t ws_bytes = 0;
  qe::DevState* st = nullptr;
  uint32_t commits = 0;  // eager mode: what DevState::commits has come to when all that was issued has run
  float* hist = nullptr;
  uint8_t* Wq = nullptr;
  uint8_t *x_stage = nullptr, *dx_stage = nullptr, *y_stage = nullptr, *dy_stage = nullptr;  // host_io only
  uint8_t *Xq[QE_MAX_SLOTS], *Gq[QE_MAX_SLOTS];
  // tensor maps over all slots (A and B roles: a_map_of, tile widths): forward, input gradient, weight gradient (MN-major)
  CUtensorMap tmXq_A[2], tmWq_B[qe::kNumTileWidths], tmGq_A[2], tmWq_dI[qe::kNumTileWidths], tmGq_dW[2], tmXq_dW[qe::kNumTileWidths];
  ActionGraph gF[QE_MAX_SLOTS], gDI[QE_MAX_SLOTS], gDW[QE_MAX_SLOTS], gDWs[QE_MAX_SLOTS], gRefresh, gCommit;
  // QE_CTX_OVERLAP_DW: per slot, "dI of the tape in this slot has been enqueued" / "the dW that released it has"
  cudaEvent_t ev_di[QE_MAX_SLOTS] = {}, ev_dw[QE_MAX_SLOTS] = {};
  bool dw_pending[QE_MAX_SLOTS] = {};
};

namespace qe_impl {

void destroy_graph(ActionGraph* g);
void ctx_release(qe_ctx* c);

// ---- execution layer
cudaError_t launch_pdl(const qe::Launch& l, cudaStream_t stream);
int32_t launch_on(const qe::Launch& l, cudaStream_t s);
int32_t launch_eager(qe_ctx* ctx, const qe::Launch& l, cudaStream_t stream);
int32_t build_graph(qe_ctx* ctx, ActionGraph* g, const std::vector<qe::Launch>& ls, cudaStream_t stream);
int32_t replay_graph(qe_ctx* ctx, ActionGraph* g, const std::vector<qe::Launch>& ls, cudaStream_t stream);
int32_t handoff_in(qe_ctx* ctx, cudaStream_t caller);
int32_t handoff_out(qe_ctx* ctx, cudaStream_t caller);
// The handshake around a call's work.  A call that an error ends in between may have kernels and copies of its own in
// flight: the caller's stream is ordered after those as well, and the error that ended the call stays the one reported.
class Handshake {
 public:
  Handshake(qe_ctx* ctx, cudaStream_t caller) : ctx_(ctx), caller_(caller) {}
  Handshake(const Handshake&) = delete;
  ~Handshake() {
    if (open_ && caller_ != ctx_->exec_stream && !ctx_->one_way && cudaEventRecord(ctx_->ev_out, ctx_->exec_stream) == cudaSuccess)
      cudaStreamWaitEvent(caller_, ctx_->ev_out, 0);
  }
  int32_t in() {
    const int32_t st = handoff_in(ctx_, caller_);
    open_ = st == QE_OK;
    return st;
  }
  int32_t out() {
    open_ = false;
    return handoff_out(ctx_, caller_);
  }

 private:
  qe_ctx* ctx_;
  cudaStream_t caller_;
  bool open_ = false;
};
int32_t host_upload(qe_ctx* ctx, void* dst, const void* src_host, size_t bytes, cudaStream_t caller);
int32_t host_download(qe_ctx* ctx, void* dst_host, const void* src, size_t bytes);
uint32_t host_pieces(uint32_t rows, const void* in, uint64_t in_bytes, const void* out, uint64_t out_bytes);
int32_t run_host_pieces(qe_layer* L, uint32_t kind, uint32_t p, uint32_t pieces, const void* in_host, void* out_host, cudaStream_t caller);
int32_t run_action(qe_ctx* ctx, ActionGraph* g, const std::vector<qe::Launch>& ls, cudaStream_t stream = nullptr);
ActionGraph* keyed_graph(qe_ctx* ctx, uint64_t key, size_t n_launches);
int32_t run_keyed(qe_ctx* ctx, uint64_t key, const std::vector<qe::Launch>& ls);

// ---- workspace and launch builders
struct Carve {
  uint64_t hist, Wq, slot0, per_slot, xq, gq, total, stage_tk = 0, stage_tn = 0;
};
Carve carve(const qe_layer_config& c);
int32_t check_config(const qe_layer_config* c);
qe::CommitParams commit_params(qe_layer* L, uint32_t mask, uint32_t bump, const float* override_amax);
qe::QuantParams quant_params(qe_layer* L, const void* x, uint8_t* q, uint32_t rows, uint32_t cols, int cls,
                             float* sinv_dst, int fmt, uint32_t commit_mask = 0);
qe::Launch quant_launch(qe_layer* L, const void* x, uint8_t* q, uint32_t rows, uint32_t cols, int cls,
                        float* sinv_dst, int fmt, uint32_t commit_mask = 0);
qe::QuantParams refresh_params(qe_layer* L);
void add_refresh(qe_layer* L, std::vector<qe::Launch>& ls);
void add_forward(qe_layer* L, uint32_t p, const void* x, void* y, std::vector<qe::Launch>& ls, qe_layer* next = nullptr,
                 uint32_t pn = 0, qe::GemmDesc* gemm_out = nullptr, qe::QuantParams* cast_out = nullptr);
void add_dI(qe_layer* L, uint32_t p, const void* dy, void* dx, std::vector<qe::Launch>& ls, qe_layer* prev = nullptr,
            uint32_t pp = 0, qe::GemmDesc* gemm_out = nullptr, qe::QuantParams* cast_out = nullptr);
qe::GemmDesc dW_gemm(qe_layer* L, uint32_t p, float* dst, int32_t accumulate, float* temp, bool sum = false);
qe::GemmDesc dW_gemm_view(qe_layer* L, uint32_t p, void* view);
void add_dW(qe_layer* L, uint32_t p, float* dst, int32_t accumulate, float* temp, std::vector<qe::Launch>& ls);

// Weight-gradient GEMMs of different layers that follow one another share one launch where the kernel allows it
// (all of whole 256-row tiles): the persistent CTAs pack their tiles into common waves and the launch is paid once.
// The layers' gradient slices are disjoint (destination registry), so the GEMMs are independent.
// Up to eight layers go out four to a launch.  More go out sixteen to a launch: sixteen 1024 x 1024 gradients of 512 tokens
// in four launches of 64 tiles leave CTA pairs idle and pay four starts and four last epilogues (chain of sixteen:
// 2397 us a step in fours, 2316 in eights, 2304 in sixteens).  One call, accumulating, sixteen to a launch against fours:
// nine of 1024 x 1024 35 us for 44, sixteen of 2048 x 2048 138 for 158 (2048 tokens: 182 for 197), twelve and sixteen of
// 4096 x 4096 334 and 443 for 334 and 445 (446 and 596 for 450 and 601).  Sixteens are faster at five to eight layers
// too (five of 1024 x 1024 30 for 33, eight of 2048 x 2048 76 for 86, eight of 4096 x 4096 at 2048 tokens 288 for 300).
struct DWBatch {
  uint32_t limit;
  std::vector<qe::GemmDesc> gp;
  std::vector<qe_layer*> layer;
  explicit DWBatch(uint32_t n_layers) : limit(n_layers > 8 ? QE_MAX_MULTI_DW : 4) {}
  bool has(const qe_layer* L) const { return std::find(layer.begin(), layer.end(), L) != layer.end(); }
  void flush(qe_ctx* ctx, std::vector<qe::Launch>& ls) {
    std::vector<qe::GemmDesc> paired;
    for (const qe::GemmDesc& g : gp)
      if (qe::whole_row_tiles(g.M)) paired.push_back(g);
    qe::Launch l;
    const bool grouped = paired.size() >= 2 && qe::make_gemm_group(paired.data(), (uint32_t)paired.size(), ctx->dev->num_sms, &l);
    if (grouped) {
      ls.push_back(l);
      ctx->stats.grouped_dw += paired.size();
    }
    for (const qe::GemmDesc& g : gp)
      if (!grouped || !qe::whole_row_tiles(g.M)) ls.push_back(qe::make_gemm(g, ctx->dev->num_sms));
    gp.clear();
    layer.clear();
  }
  void add(qe_ctx* ctx, qe_layer* L, const qe::GemmDesc& g, std::vector<qe::Launch>& ls) {
    if (gp.size() == limit || has(L)) flush(ctx, ls);  // a layer's own GEMMs accumulate into one slice: never in one launch
    gp.push_back(g);
    layer.push_back(L);
  }
};

struct Fnv {
  uint64_t key = 1469598103934665603ull;  // FNV-1a
  void mix(const void* ptr, size_t n) {
    const unsigned char* c = (const unsigned char*)ptr;
    for (size_t i = 0; i < n; ++i) key = (key ^ c[i]) * 1099511628211ull;
  }
};


}  // namespace qe_impl
