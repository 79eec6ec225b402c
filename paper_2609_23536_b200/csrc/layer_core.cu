// Execution layer and launch builders of the layer API (definitions of layer_impl.h).
#include "layer_impl.h"

namespace qe_impl {

DeviceInfo g_dev[16];

// Per-device one-time setup: SM count, compute capability, driver entry point for tensor-map encoding, and the
// GEMM's shared-memory opt-in.  The device must be current.
int32_t device_info(int device, DeviceInfo** out) {
  if (device < 0 || device >= 16) return fail(QE_ERR_BAD_ARG, "device %d", device);
  DeviceInfo& d = g_dev[device];
  if (!d.ready) {
    cudaDeviceProp prop;
    QE_CUDA(cudaGetDeviceProperties(&prop, device));
    if (prop.major != 10) return fail(QE_ERR_UNSUPPORTED, "device %d is sm_%d%d; this library needs sm_100", device, prop.major, prop.minor);
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult qres;
    QE_CUDA(cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres));
    if (!fn || qres != cudaDriverEntryPointSuccess) return fail(QE_ERR_CUDA, "cuTensorMapEncodeTiled not available");
    QE_CUDA(qe::gemm_prepare());
    d.device = device;
    d.num_sms = prop.multiProcessorCount;
    d.cc_major = prop.major;
    d.encode = (EncodeTiledFn)fn;
    d.ready = true;
  }
  *out = &d;
  return QE_OK;
}

// Tensor map over a GEMM operand of `rows` rows: contraction-major bytes [rows, Kc], or (mn) [Kc, rows].  Its box holds box_rows
// (128, 64 or 32) rows of `blocks` K blocks of 128, one block behind the other: dimensions (byte of the block, row, block) or
// (row, K row of the block, block), and the tensor's number among those of the same shape that follow at `apart` bytes.  128
// contraction bytes (mn: box_rows bytes) lie together, swizzled over that length.
int32_t make_map(const DeviceInfo* d, CUtensorMap* map, const Slots& t, uint64_t rows, uint64_t Kc, bool mn, uint32_t box_rows,
                 uint32_t blocks) {
  cuuint64_t gdim[4] = {mn ? rows : 128u, mn ? 128u : rows, Kc / 128u, t.count};
  cuuint64_t gstride[3] = {mn ? rows : Kc, mn ? 128u * rows : 128u, t.count > 1 ? t.apart : rows * Kc};
  cuuint32_t box[4] = {mn ? box_rows : 128u, mn ? 128u : box_rows, blocks, 1u};
  cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  const CUtensorMapSwizzle sw = box[0] == 128u ? CU_TENSOR_MAP_SWIZZLE_128B : box[0] == 64u ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B;
  CUresult r = d->encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 4, const_cast<void*>(t.first), gdim, gstride, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(QE_ERR_CUDA, "cuTensorMapEncodeTiled failed with %d", (int)r);
  return QE_OK;
}

// The map of a GEMM's A operand for launches of one tile width, or of its B operand.
int32_t make_a_map(const DeviceInfo* d, CUtensorMap* map, const Slots& t, uint64_t M, uint64_t Kc, bool mn, uint32_t width) {
  return make_map(d, map, t, M, Kc, mn, 128, qe::blocks_of(width));
}
int32_t make_b_map(const DeviceInfo* d, CUtensorMap* map, const Slots& t, uint64_t N, uint64_t Kc, bool mn, uint32_t width) {
  return make_map(d, map, t, N, Kc, mn, qe::kTileWidths[width] / 2, qe::blocks_of(width));
}
// ... for all of them: operands that a layer keeps.
int32_t make_a_maps(const DeviceInfo* d, CUtensorMap* maps, const Slots& t, uint64_t M, uint64_t Kc, bool mn) {
  for (uint32_t w = 0; w < 2; ++w) {
    const int32_t st = make_a_map(d, &maps[qe::a_map_of(w)], t, M, Kc, mn, w);
    if (st != QE_OK) return st;
  }
  return QE_OK;
}
int32_t make_b_maps(const DeviceInfo* d, CUtensorMap* maps, const Slots& t, uint64_t N, uint64_t Kc, bool mn) {
  for (uint32_t w = 0; w < qe::kNumTileWidths; ++w) {
    const int32_t st = make_b_map(d, &maps[w], t, N, Kc, mn, w);
    if (st != QE_OK) return st;
  }
  return QE_OK;
}

// Tensor map over the output D [M, N] (row pitch ldo elements) for the epilogue's bulk stores: boxes of 32 columns and 32 rows
// (FP32 sums of products: 128); bf16 rows of a box are 64 bytes (64-byte swizzle), FP32 rows 128 bytes (128-byte swizzle).
int32_t make_out_map(const DeviceInfo* d, CUtensorMap* map, const void* ptr, uint64_t M, uint64_t N, uint64_t ldo,
                     bool fp32, uint32_t rows) {
  cuuint64_t gdim[2] = {N, M};
  cuuint64_t gstride[1] = {ldo * (fp32 ? 4u : 2u)};
  cuuint32_t box[2] = {32u, rows};
  cuuint32_t estr[2] = {1u, 1u};
  CUresult r = d->encode(map, fp32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2,
                         const_cast<void*>(ptr), gdim, gstride, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         fp32 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(QE_ERR_CUDA, "cuTensorMapEncodeTiled (output) failed with %d", (int)r);
  return QE_OK;
}

// Tensor map over FP8 bytes D [M, N] (row pitch ld bytes) for the hand-off epilogue: 32-byte x 32-row boxes, no swizzle.
int32_t make_out_map_u8(const DeviceInfo* d, CUtensorMap* map, const void* ptr, uint64_t M, uint64_t N, uint64_t ld) {
  cuuint64_t gdim[2] = {N, M};
  cuuint64_t gstride[1] = {ld};
  cuuint32_t box[2] = {32u, 32u};
  cuuint32_t estr[2] = {1u, 1u};
  CUresult r = d->encode(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(ptr), gdim, gstride, box, estr,
                         CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                         CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(QE_ERR_CUDA, "cuTensorMapEncodeTiled (FP8 output) failed with %d", (int)r);
  return QE_OK;
}


int32_t current_device_info(DeviceInfo** d) {
  int dev = 0;
  QE_CUDA(cudaGetDevice(&dev));
  return device_info(dev, d);
}

int32_t launch_on(const qe::Launch& l, cudaStream_t s) {
  QE_CUDA(launch_pdl(l, s));
  return QE_OK;
}


void destroy_graph(ActionGraph* g) {
  if (g->exec) cudaGraphExecDestroy(g->exec);
  if (g->graph) cudaGraphDestroy(g->graph);
  g->exec = nullptr;
  g->graph = nullptr;
  g->built = false;
}
void ctx_release(qe_ctx* c) {
  if (!c->closed || c->layers) return;
  cudaStreamSynchronize(c->exec_stream);
  for (auto* sg : c->step_graphs) {
    destroy_graph(&sg->g);
    delete sg;
  }
  if (c->dw_stream) {
    cudaStreamSynchronize(c->dw_stream);
    cudaStreamDestroy(c->dw_stream);
    cudaEventDestroy(c->ev_dw_in);
  }
  if (c->h2d_stream) {
    cudaStreamSynchronize(c->h2d_stream);
    cudaStreamSynchronize(c->d2h_stream);
    cudaStreamDestroy(c->h2d_stream);
    cudaStreamDestroy(c->d2h_stream);
    cudaEventDestroy(c->ev_h2d);
    cudaEventDestroy(c->ev_kernels);
    cudaEventDestroy(c->ev_d2h);
  }
  cudaEventDestroy(c->ev_in);
  cudaEventDestroy(c->ev_out);
  if (c->owns_stream) cudaStreamDestroy(c->exec_stream);
  qe_registry_destroy(c->registry);
  delete c;
}



// One launch with programmatic stream serialization: the kernel may be scheduled while its predecessor in the stream
// drains; every kernel of the library waits for its predecessors (griddepcontrol.wait) before touching their data, or, a
// cast that may overlap a GEMM launch, acquires that launch's commits (Announce).
cudaError_t launch_pdl(const qe::Launch& l, cudaStream_t stream) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = l.grid;
  cfg.blockDim = l.block;
  cfg.dynamicSmemBytes = l.smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeCooperative;
  attr[1].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = l.cooperative ? 2 : 1;
  qe::Launch::Block tmp;
  void* args[1] = {l.args_block(&tmp)};
  return cudaLaunchKernelExC(&cfg, l.func, args);
}

int32_t launch_eager(qe_ctx* ctx, const qe::Launch& l, cudaStream_t stream) {
  QE_CUDA(launch_pdl(l, stream));
  ctx->stats.eager_launches += 1;
  ctx->stats.kernels_launched += 1;
  return QE_OK;
}

// Capture the launches on the execution stream into a graph, instantiate it, and recover the kernel nodes in
// launch order by walking the (linear) dependency chain from the root.
int32_t build_graph(qe_ctx* ctx, ActionGraph* g, const std::vector<qe::Launch>& ls, cudaStream_t stream) {
  const auto t0 = std::chrono::steady_clock::now();
  std::vector<qe::Launch> kept = ls;  // (all memory before the capture: nothing below fails for lack of it)
  std::vector<cudaGraphNode_t> chain;
  chain.reserve(ls.size());
  QE_CUDA(cudaStreamBeginCapture(stream, cudaStreamCaptureModeThreadLocal));
  cudaError_t err = cudaSuccess;
  for (const qe::Launch& l : ls) {
    err = launch_pdl(l, stream);
    if (err != cudaSuccess) break;
  }
  cudaGraph_t graph = nullptr;
  cudaError_t end = cudaStreamEndCapture(stream, &graph);
  if (err != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    return fail(QE_ERR_CUDA, "launch during capture: %s", cudaGetErrorString(err));
  }
  QE_CUDA(end);
  size_t n = 0;
  QE_CUDA(cudaGraphGetNodes(graph, nullptr, &n));
  if (n != ls.size()) {
    cudaGraphDestroy(graph);
    return fail(QE_ERR_CUDA, "captured %zu nodes for %zu launches", n, ls.size());
  }
  size_t nroot = 1;
  cudaGraphNode_t cur = nullptr;
  QE_CUDA(cudaGraphGetRootNodes(graph, &cur, &nroot));
  if (nroot != 1) {
    cudaGraphDestroy(graph);
    return fail(QE_ERR_CUDA, "captured graph has %zu roots", nroot);
  }
  while (cur) {
    chain.push_back(cur);
    // the edges carry programmatic-dependency data, which only the _v2 query reports
    size_t nd = 0;
    QE_CUDA(cudaGraphNodeGetDependentNodes_v2(cur, nullptr, nullptr, &nd));
    if (nd == 0) break;
    if (nd != 1) return fail(QE_ERR_CUDA, "captured graph is not a chain");
    cudaGraphNode_t next = nullptr;
    cudaGraphEdgeData edge{};
    QE_CUDA(cudaGraphNodeGetDependentNodes_v2(cur, &next, &edge, &nd));
    cur = next;
  }
  if (chain.size() != ls.size()) {
    cudaGraphDestroy(graph);
    return fail(QE_ERR_CUDA, "chain of %zu nodes for %zu launches", chain.size(), ls.size());
  }
  cudaGraphExec_t exec = nullptr;
  cudaError_t ie = cudaGraphInstantiate(&exec, graph, 0);
  if (ie != cudaSuccess) {
    cudaGraphDestroy(graph);
    return fail(QE_ERR_CUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(ie));
  }
  g->graph = graph;
  g->exec = exec;
  g->nodes = std::move(chain);
  g->launches = std::move(kept);
  g->built = true;
  ctx->stats.graphs_built += 1;
  ctx->stats.capture_host_ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  return QE_OK;
}

int32_t replay_graph(qe_ctx* ctx, ActionGraph* g, const std::vector<qe::Launch>& ls, cudaStream_t stream) {
  if (ls.size() != g->launches.size()) return fail(QE_ERR_CUDA, "graph shape changed");
  for (size_t i = 0; i < ls.size(); ++i) {
    const qe::Launch& now = ls[i];
    qe::Launch& was = g->launches[i];
    const bool same = now.func == was.func && now.params.size() == was.params.size() && now.smem == was.smem &&
                      now.grid.x == was.grid.x && now.grid.y == was.grid.y && now.block.x == was.block.x &&
                      std::memcmp(now.params.data(), was.params.data(), now.params.size()) == 0;
    if (same) continue;
    // caller-visible pointers (x, y, gradient destination) or the accumulate flag changed: patch the node in place
    cudaKernelNodeParams np{};
    qe::Launch::Block tmp;
    void* args[1] = {now.args_block(&tmp)};
    np.func = const_cast<void*>(now.func);
    np.gridDim = now.grid;
    np.blockDim = now.block;
    np.sharedMemBytes = now.smem;
    np.kernelParams = args;
    np.extra = nullptr;
    QE_CUDA(cudaGraphExecKernelNodeSetParams(g->exec, g->nodes[i], &np));
    was = now;
    ctx->stats.node_param_updates += 1;
  }
  QE_CUDA(cudaGraphLaunch(g->exec, stream));
  ctx->stats.graph_replays += 1;
  ctx->stats.kernels_launched += ls.size();
  return QE_OK;
}

// Sec. 4.4: the execution stream waits on the caller's stream before the action...
int32_t handoff_in(qe_ctx* ctx, cudaStream_t caller) {
  if (caller == ctx->exec_stream) return QE_OK;
  QE_CUDA(cudaEventRecord(ctx->ev_in, caller));
  QE_CUDA(cudaStreamWaitEvent(ctx->exec_stream, ctx->ev_in, 0));
  ctx->stats.handoffs += 1;
  return QE_OK;
}
// ...and the caller's stream waits on the action's tail before it may consume anything.
int32_t handoff_out(qe_ctx* ctx, cudaStream_t caller) {
  if (caller == ctx->exec_stream) return QE_OK;
  if (ctx->one_way) return QE_OK;  // the defective protocol, kept for the stale-read experiment only
  QE_CUDA(cudaEventRecord(ctx->ev_out, ctx->exec_stream));
  QE_CUDA(cudaStreamWaitEvent(caller, ctx->ev_out, 0));
  ctx->stats.handoffs += 1;
  return QE_OK;
}

// ---- host-buffer calls.  The upload of an action runs on one copy stream and the read-back of its result on
// another, so that the upload of action k+1 overlaps the read-back of action k (the host link is full duplex); the
// kernels stay on the execution stream, which waits for the upload before them and for the read-back after them
// (a caller that synchronises after the call finds its host buffer complete).  An upload comes after every earlier
// read-back that writes what it reads.
static int32_t uploads_after_readbacks(qe_ctx* ctx) {
  QE_CUDA(cudaStreamWaitEvent(ctx->h2d_stream, ctx->ev_d2h, 0));  // recorded after the latest of them
  ctx->readbacks.clear();
  return QE_OK;
}

// Before a call's uploads from [src_host, src_host + bytes).
static int32_t uploads_begin(qe_ctx* ctx, const void* src_host, size_t bytes, cudaStream_t caller) {
  if (!ctx->h2d_stream) {
    ctx->readbacks.reserve(256);
    cudaError_t e = cudaStreamCreateWithFlags(&ctx->h2d_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&ctx->d2h_stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ev_h2d, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ev_kernels, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ctx->ev_d2h, cudaEventDisableTiming);
    if (e != cudaSuccess) return fail(QE_ERR_CUDA, "copy streams: %s", cudaGetErrorString(e));
  }
  // the staging buffer was last read by the kernels of an earlier host-buffer call
  if (ctx->kernels_recorded) QE_CUDA(cudaStreamWaitEvent(ctx->h2d_stream, ctx->ev_kernels, 0));
  if (caller != ctx->exec_stream) {
    QE_CUDA(cudaStreamWaitEvent(ctx->h2d_stream, ctx->ev_in, 0));  // recorded by handoff_in, after the read-backs of earlier calls
  } else {
    // (the execution stream itself: waiting for all of it would keep uploads and read-backs from overlapping)
    const uintptr_t lo = (uintptr_t)src_host, hi = lo + bytes;
    for (const qe_ctx::HostRange& r : ctx->readbacks)
      if (r.lo < hi && lo < r.hi) {
        const int32_t st = uploads_after_readbacks(ctx);
        if (st != QE_OK) return st;
        break;
      }
  }
  return QE_OK;
}
// One upload; the kernels that follow wait for it.
static int32_t upload(qe_ctx* ctx, void* dst, const void* src_host, size_t bytes) {
  QE_CUDA(cudaMemcpyAsync(dst, src_host, bytes, cudaMemcpyHostToDevice, ctx->h2d_stream));
  QE_CUDA(cudaEventRecord(ctx->ev_h2d, ctx->h2d_stream));
  QE_CUDA(cudaStreamWaitEvent(ctx->exec_stream, ctx->ev_h2d, 0));
  return QE_OK;
}
int32_t host_upload(qe_ctx* ctx, void* dst, const void* src_host, size_t bytes, cudaStream_t caller) {
  const int32_t st = uploads_begin(ctx, src_host, bytes, caller);
  return st != QE_OK ? st : upload(ctx, dst, src_host, bytes);
}
// After kernels: frees what they read for the next upload and starts the read-back of what they wrote (if any).
static int32_t download(qe_ctx* ctx, void* dst_host, const void* src, size_t bytes) {
  QE_CUDA(cudaEventRecord(ctx->ev_kernels, ctx->exec_stream));
  ctx->kernels_recorded = true;
  if (!dst_host) return QE_OK;
  const uintptr_t lo = (uintptr_t)dst_host;
  if (!ctx->readbacks.empty() && ctx->readbacks.back().hi == lo) {
    ctx->readbacks.back().hi += bytes;  // a call's next piece
  } else {
    if (ctx->readbacks.size() == 256) {
      const int32_t st = uploads_after_readbacks(ctx);
      if (st != QE_OK) return st;
    }
    ctx->readbacks.push_back({lo, lo + bytes});
  }
  QE_CUDA(cudaStreamWaitEvent(ctx->d2h_stream, ctx->ev_kernels, 0));
  QE_CUDA(cudaMemcpyAsync(dst_host, src, bytes, cudaMemcpyDeviceToHost, ctx->d2h_stream));
  QE_CUDA(cudaEventRecord(ctx->ev_d2h, ctx->d2h_stream));
  return QE_OK;
}
// After a call's last read-back: what the execution stream is given next comes after it.
static int32_t downloads_end(qe_ctx* ctx, const void* dst_host) {
  if (dst_host) QE_CUDA(cudaStreamWaitEvent(ctx->exec_stream, ctx->ev_d2h, 0));
  return QE_OK;
}
int32_t host_download(qe_ctx* ctx, void* dst_host, const void* src, size_t bytes) {
  const int32_t st = download(ctx, dst_host, src, bytes);
  return st != QE_OK ? st : downloads_end(ctx, dst_host);
}

// Whether copies from or to host memory run beside the host.
static bool pinned(const void* p) {
  cudaPointerAttributes a{};
  if (cudaPointerGetAttributes(&a, p) == cudaSuccess) return a.type != cudaMemoryTypeUnregistered;
  cudaGetLastError();  // (the question's, not a call's)
  return false;
}

// Pieces of rows in which a forward or an input gradient with host buffers goes through upload, kernels and read-back: the
// host link carries both directions at once, but one after the other a call's input, kernels and output used it one at a time.
// Two pieces, or one for every 512 rows up to four, of whole 256-row tiles, whose larger copy is a megabyte at least (19 us at 53
// GB/s; a piece costs some 15 us of copy starts, events and kernels that its neighbours' copies have to cover).  us a step in one
// piece / two / up to four of 256 rows: a block of hidden 1024, 1024 tokens, 6385 / 5716 / 5861; 2048 tokens, 1024 x 3072 and
// 1024 x 1024, 3252 / 2949 / 2882; 640 tokens, 2048 x 2048 and 2048 x 512, 1377 / 1313 / 1312; up to eight of 128 rows 6428 and 3152.  In one
// piece / four: 4096 tokens, 1024 x 3072 and 1024 x 1024, 4018 / 3503, 4096 x 4096 5286 / 3927; 8192, 2048 x 2048 and 2048 x 512, 8375 / 6665.
// An output that overlaps the input is read back when all of that has been uploaded.  Pageable memory goes through in one piece:
// each of its copies is over before the call goes on, so that pieces would only add waits (F and dI of 1024 x 3072 at 1024 tokens
// 1050 us in one, 1220 in two; 2048 x 2048 at 2048 tokens 1900 and 2380, at 4096 3580 and 4270 in four).
uint32_t host_pieces(uint32_t rows, const void* in, uint64_t in_bytes, const void* out, uint64_t out_bytes) {
  if (!out) out_bytes = 0;
  if ((uintptr_t)in < (uintptr_t)out + out_bytes && (uintptr_t)out < (uintptr_t)in + in_bytes) return 1;
  const uint64_t most = std::min<uint64_t>(4, std::max<uint64_t>(2, rows / 512u));
  const uint64_t n = std::min<uint64_t>({most, rows / 256u, std::max(in_bytes, out_bytes) >> 20});
  return n > 1 && pinned(in) && (!out || pinned(out)) ? (uint32_t)n : 1u;
}

// F (kind QE_ACT_F) or dI of slot p with host buffers, in pieces; the scale commits go with the last piece's GEMM, whose launch
// starts after every piece's cast.  All launches are made before the first kernel and the first read-back go out: what can fail for
// want of memory fails with nothing but an upload on its way.
int32_t run_host_pieces(qe_layer* L, uint32_t kind, uint32_t p, uint32_t pieces, const void* in_host, void* out_host, cudaStream_t caller) {
  qe_ctx* ctx = L->ctx;
  const uint32_t T = L->cfg.T, cols_in = kind == QE_ACT_F ? L->cfg.K : L->cfg.N, cols_out = kind == QE_ACT_F ? L->cfg.N : L->cfg.K;
  uint8_t* const in = kind == QE_ACT_F ? L->x_stage : L->dy_stage;
  uint8_t* const out = kind == QE_ACT_F ? L->y_stage : L->dx_stage;
  uint8_t* const q = kind == QE_ACT_F ? L->Xq[p] : L->Gq[p];
  const uint32_t share = T / pieces / 256u * 256u;
  const auto first_row = [&](uint32_t i) { return i < pieces ? i * share : T; };
  const auto upload_piece = [&](uint32_t i) {
    const size_t at = 2ull * first_row(i) * cols_in;
    return upload(ctx, in + at, (const uint8_t*)in_host + at, 2ull * first_row(i + 1) * cols_in - at);
  };
  int32_t st = uploads_begin(ctx, in_host, 2ull * T * cols_in, caller);
  if (st == QE_OK) st = upload_piece(0);
  if (st != QE_OK) return st;
  std::vector<qe::Launch> ls;
  ls.reserve(2 * pieces);
  for (uint32_t i = 0; i < pieces; ++i) {
    const uint32_t row0 = first_row(i), rows = first_row(i + 1) - row0;
    qe::GemmDesc g;
    qe::QuantParams cast;
    if (kind == QE_ACT_F) add_forward(L, p, in + 2ull * row0 * cols_in, out + 2ull * row0 * cols_out, ls, nullptr, 0, &g, &cast);
    else add_dI(L, p, in + 2ull * row0 * cols_in, out + 2ull * row0 * cols_out, ls, nullptr, 0, &g, &cast);
    cast.q += (size_t)row0 * cols_in;
    cast.rows = rows;
    CUtensorMap map[2];  // of this piece's rows
    if ((st = make_a_maps(ctx->dev, map, Slots{q + (size_t)row0 * cols_in}, rows, cols_in, false)) != QE_OK) return st;
    if ((st = make_out_map(ctx->dev, &g.tmD, g.out, rows, cols_out, cols_out, false)) != QE_OK) return st;
    g.M = rows;
    g.operands(map, &g.alpha_a[p], 0, g.mapB, g.alpha_b, 0);
    if (i + 1 < pieces) g.commit = qe::CommitParams{};
    ls.push_back(qe::make_quantize(cast));
    ls.push_back(qe::make_gemm(g, ctx->dev->num_sms));
  }
  for (uint32_t i = 0; i < pieces && st == QE_OK; ++i) {
    if (i) st = upload_piece(i);
    for (uint32_t k = 2 * i; k < 2 * i + 2 && st == QE_OK; ++k)  // (no graph: a piece's two launches hide behind the copies, and a
      st = launch_eager(ctx, ls[k], ctx->exec_stream);           // new layer has none to make)
    const size_t at = 2ull * first_row(i) * cols_out;
    if (st == QE_OK) st = download(ctx, out_host ? (uint8_t*)out_host + at : nullptr, out + at, 2ull * first_row(i + 1) * cols_out - at);
  }
  const int32_t end = downloads_end(ctx, out_host);  // (also when a piece failed: read-backs may be on their way)
  return st != QE_OK ? st : end;
}

int32_t run_action(qe_ctx* ctx, ActionGraph* g, const std::vector<qe::Launch>& ls, cudaStream_t stream) {
  if (!stream) stream = ctx->exec_stream;
  if (ctx->exec_mode == QE_EXEC_GRAPH) {
    if (!g->built) {
      int32_t st = build_graph(ctx, g, ls, stream);
      if (st != QE_OK) return st;
    }
    return replay_graph(ctx, g, ls, stream);
  }
  for (const qe::Launch& l : ls) {
    int32_t st = launch_eager(ctx, l, stream);
    if (st != QE_OK) return st;
  }
  return QE_OK;
}

// Graph of a launch list identified by a hash (whole steps, multi-layer dW calls); rebuilt when the list's length
// changed under the same key (e.g. no weight refresh this time).
ActionGraph* keyed_graph(qe_ctx* ctx, uint64_t key, size_t n_launches) {
  qe_ctx::StepGraph* sg = nullptr;
  for (auto* c : ctx->step_graphs)
    if (c->key == key) sg = c;
  if (sg && sg->g.launches.size() != n_launches) {
    destroy_graph(&sg->g);
    sg->g = ActionGraph();
  }
  if (!sg) {
    ctx->step_graphs.reserve(ctx->step_graphs.size() + 1);
    sg = new (std::nothrow) qe_ctx::StepGraph();
    if (!sg) return nullptr;
    sg->key = key;
    ctx->step_graphs.push_back(sg);
  }
  return &sg->g;
}


int32_t run_keyed(qe_ctx* ctx, uint64_t key, const std::vector<qe::Launch>& ls) {
  if (ctx->exec_mode == QE_EXEC_GRAPH) {
    ActionGraph* g = keyed_graph(ctx, key, ls.size());
    if (!g) return fail(QE_ERR_BAD_ARG, "out of host memory");
    return run_action(ctx, g, ls);
  }
  for (const qe::Launch& l : ls) {
    int32_t st = launch_eager(ctx, l, ctx->exec_stream);
    if (st != QE_OK) return st;
  }
  return QE_OK;
}




Carve carve(const qe_layer_config& c) {
  Carve k{};
  uint64_t o = sizeof(qe::DevState);
  k.hist = o;
  o = align_up(o + 4ull * c.history_len * sizeof(float), 1024);
  const uint64_t nk = (uint64_t)c.N * c.K, tk = (uint64_t)c.T * c.K, tn = (uint64_t)c.T * c.N;
  // One FP8 copy of every tensor, row-major: the GEMMs read it contraction-major or MN-major, as each of them needs.
  k.Wq = o;
  o += align_up(nk, 1024);
  k.slot0 = o;
  k.xq = 0;
  k.gq = align_up(tk, 1024);
  k.per_slot = k.gq + align_up(tn, 1024);
  o += k.per_slot * c.slots;
  if (c.host_io) {  // x / dx [T,K] and y / dy [T,N] bf16 staging for the host-buffer entry points
    k.stage_tk = o;
    o += 2 * align_up(2 * tk, 1024);
    k.stage_tn = o;
    o += 2 * align_up(2 * tn, 1024);
  }
  k.total = o;
  return k;
}

int32_t check_config(const qe_layer_config* c) {
  if (!c) return fail(QE_ERR_BAD_ARG, "config is null");
  if (!shape_ok(c->T) || !shape_ok(c->K) || !shape_ok(c->N))
    return fail(QE_ERR_SHAPE, "T=%u K=%u N=%u: each must be a multiple of 128 in [256, 2^20]", c->T, c->K, c->N);
  if (c->history_len < 1 || c->history_len > QE_MAX_HISTORY) return fail(QE_ERR_BAD_ARG, "history_len %u", c->history_len);
  if (c->margin < -32 || c->margin > 32) return fail(QE_ERR_BAD_ARG, "margin %d", c->margin);
  if (c->slots < 1 || c->slots > QE_MAX_SLOTS) return fail(QE_ERR_BAD_ARG, "slots %u", c->slots);
  if (c->host_io > 1) return fail(QE_ERR_BAD_ARG, "host_io %u", c->host_io);
  return QE_OK;
}

qe::CommitParams commit_params(qe_layer* L, uint32_t mask, uint32_t bump, const float* override_amax) {
  qe::CommitParams cp{};
  cp.st = L->st;
  cp.hist = L->hist;
  cp.H = L->cfg.history_len;
  cp.class_mask = mask;
  cp.pow2_neg_margin = std::ldexp(1.0f, -L->cfg.margin);
  cp.amax_override = override_amax;
  cp.bump_token = bump;
  return cp;
}

// commit_mask != 0: the kernel's last block also commits those classes (used for the weight refresh)
qe::QuantParams quant_params(qe_layer* L, const void* x, uint8_t* q, uint32_t rows, uint32_t cols, int cls,
                             float* sinv_dst, int fmt, uint32_t commit_mask) {
  qe::QuantParams qp{};
  qp.x = (const uint16_t*)x;
  qp.q = q;
  qp.rows = rows;
  qp.cols = cols;
  qp.scale = &L->st->scale[cls];
  qp.sinv_src = &L->st->scale_inv[cls];
  qp.sinv_dst = sinv_dst;
  qp.amax_bits = &L->st->pending_amax[cls];
  qp.fmt = fmt;
  if (commit_mask) qp.commit = commit_params(L, commit_mask, 0, nullptr);
  return qp;
}
qe::Launch quant_launch(qe_layer* L, const void* x, uint8_t* q, uint32_t rows, uint32_t cols, int cls,
                        float* sinv_dst, int fmt, uint32_t commit_mask) {
  return qe::make_quantize(quant_params(L, x, q, rows, cols, cls, sinv_dst, fmt, commit_mask));
}


// ---- the launches of each action (shared by the per-action calls and the whole-step call)
// Invariant 3: first forward of the epoch re-quantises the weight; the kernel's last block commits its amax
qe::QuantParams refresh_params(qe_layer* L) {
  return quant_params(L, L->cfg.weight_dev, L->Wq, L->cfg.N, L->cfg.K, QE_CLASS_W, &L->st->cache_sinv_W, QE_E4M3, 1u << QE_CLASS_W);
}
void add_refresh(qe_layer* L, std::vector<qe::Launch>& ls) { ls.push_back(qe::make_quantize(refresh_params(L))); }

// FP8 hand-off between directly chained linears: the forward GEMM of `L` emits its output as the E4M3 input of
// `next` (quantised with next's current X scale, straight into next's tape slot pn, with next's X amax and
// inverse-scale snapshot), so `next` needs no cast kernel; x == null means L's own input was deposited that way.
// gemm_out != null: the GEMM is handed back instead of being queued (the caller puts it into a shared launch).
void add_forward(qe_layer* L, uint32_t p, const void* x, void* y, std::vector<qe::Launch>& ls, qe_layer* next,
                 uint32_t pn, qe::GemmDesc* gemm_out, qe::QuantParams* cast_out) {
  const uint32_t T = L->cfg.T, K = L->cfg.K, N = L->cfg.N;
  if (x && cast_out) *cast_out = quant_params(L, x, L->Xq[p], T, K, QE_CLASS_X, &L->st->slot_sinv_X[p], QE_E4M3);
  else if (x) ls.push_back(quant_launch(L, x, L->Xq[p], T, K, QE_CLASS_X, &L->st->slot_sinv_X[p], QE_E4M3));
  qe::GemmDesc own;
  qe::GemmDesc& gp = gemm_out ? *gemm_out : own;  // (as it was made: nothing set yet)
  gp.operands(L->tmXq_A, L->st->slot_sinv_X, p, L->tmWq_B, &L->st->cache_sinv_W, 0);
  gp.M = T;
  gp.N = N;
  gp.Kc = K;
  gp.a_fmt = gp.b_fmt = QE_E4M3;
  gp.ldo = N;
  if (next) {
    gp.out = next->Xq[pn];
    gp.epi = 3;
    make_out_map_u8(L->ctx->dev, &gp.tmD, next->Xq[pn], T, N, N);
    gp.out_scale = &next->st->scale[QE_CLASS_X];
    gp.out_fmt = QE_E4M3;
    gp.amax_bits2 = &next->st->pending_amax[QE_CLASS_X];
    gp.sinv_src = &next->st->scale_inv[QE_CLASS_X];
    gp.sinv_dst = &next->st->slot_sinv_X[pn];
  } else {
    gp.out = y;
    gp.epi = 0;
    make_out_map(L->ctx->dev, &gp.tmD, y, T, N, N, false);
  }
  gp.amax_bits = &L->st->pending_amax[QE_CLASS_Y];
  gp.status = &L->st->status;
  gp.commit = commit_params(L, 1u << QE_CLASS_Y, 1, nullptr);  // done by the GEMM's last CTA ...
  gp.commit.early_mask = 1u << QE_CLASS_X;                     // ... and by its first, once the cast before it is complete
  if (!gemm_out) ls.push_back(qe::make_gemm(gp, L->ctx->dev->num_sms));
}

// Hand-off in the backward direction: the input gradient of `L` is the output gradient of the linear before it
// (`prev`), emitted as E5M2 with prev's G scale into prev's tape slot pp; dy == null: L's own dY came that way.
void add_dI(qe_layer* L, uint32_t p, const void* dy, void* dx, std::vector<qe::Launch>& ls, qe_layer* prev,
            uint32_t pp, qe::GemmDesc* gemm_out, qe::QuantParams* cast_out) {
  const uint32_t T = L->cfg.T, K = L->cfg.K, N = L->cfg.N;
  if (dy && cast_out) *cast_out = quant_params(L, dy, L->Gq[p], T, N, QE_CLASS_G, &L->st->slot_sinv_G[p], QE_E5M2);
  else if (dy) ls.push_back(quant_launch(L, dy, L->Gq[p], T, N, QE_CLASS_G, &L->st->slot_sinv_G[p], QE_E5M2));
  qe::GemmDesc own;
  qe::GemmDesc& gp = gemm_out ? *gemm_out : own;  // (as it was made: nothing set yet)
  gp.operands(L->tmGq_A, L->st->slot_sinv_G, p, L->tmWq_dI, &L->st->cache_sinv_W, 0);
  gp.M = T;
  gp.N = K;
  gp.Kc = N;
  gp.a_fmt = QE_E5M2;
  gp.b_fmt = QE_E4M3;
  gp.b_mn = 1;  // Wq [N,K] itself: B in MN-major form
  gp.ldo = K;
  if (prev) {
    gp.out = prev->Gq[pp];
    gp.epi = 3;
    make_out_map_u8(L->ctx->dev, &gp.tmD, prev->Gq[pp], T, K, K);
    gp.out_scale = &prev->st->scale[QE_CLASS_G];
    gp.out_fmt = QE_E5M2;
    gp.amax_bits2 = &prev->st->pending_amax[QE_CLASS_G];
    gp.sinv_src = &prev->st->scale_inv[QE_CLASS_G];
    gp.sinv_dst = &prev->st->slot_sinv_G[pp];
  } else {
    gp.out = dx;
    gp.epi = 0;
    make_out_map(L->ctx->dev, &gp.tmD, dx, T, K, K, false);
  }
  gp.amax_bits = nullptr;
  gp.status = &L->st->status;
  gp.commit = commit_params(L, 0, 1, nullptr);  // backward amax/scale updated exactly once, here: the cast (or the
  gp.commit.early_mask = 1u << QE_CLASS_G;      // hand-off) that made Gq has completed the amax before this GEMM starts
  if (!gemm_out) ls.push_back(qe::make_gemm(gp, L->ctx->dev->num_sms));
}

// The weight-gradient GEMM of slot p; dst = first element of the layer's gradient slice, temp != null makes it
// write the temporary instead (copied-gradient comparison path); sum: products of other slots are going to be added.
qe::GemmDesc dW_gemm(qe_layer* L, uint32_t p, float* dst, int32_t accumulate, float* temp, bool sum) {
  const uint32_t T = L->cfg.T, K = L->cfg.K, N = L->cfg.N;
  qe::GemmDesc gp;
  // (scales: the snapshots taken when dY_m and X_m were quantised, never the current state)
  gp.operands(L->tmGq_dW, L->st->slot_sinv_G, p, L->tmXq_dW, L->st->slot_sinv_X, p);
  gp.M = N;
  gp.N = K;
  gp.Kc = T;
  gp.a_fmt = QE_E5M2;
  gp.b_fmt = QE_E4M3;
  gp.a_mn = gp.b_mn = 1;  // Gq [T,N] and Xq [T,K] themselves, read as MN-major operands
  gp.ldo = K;
  gp.amax_bits = nullptr;
  gp.status = &L->st->status;
  make_out_map(L->ctx->dev, &gp.tmD, temp ? temp : dst, N, K, K, true, sum ? 128 : 32);
  gp.sum = sum;
  if (!temp) {
    gp.out = dst;  // direct placement: the epilogue reads, adds and writes the destination itself
    gp.epi = accumulate ? 2 : 1;
  } else {
    gp.out = temp;
    gp.epi = 1;
  }
  return gp;
}

// Per-microbatch arena: the same GEMM writes bf16(D) into the microbatch's own view (no accumulation, no amax).
qe::GemmDesc dW_gemm_view(qe_layer* L, uint32_t p, void* view) {
  qe::GemmDesc gp = dW_gemm(L, p, nullptr, 0, nullptr);
  gp.out = view;
  gp.epi = 0;
  make_out_map(L->ctx->dev, &gp.tmD, view, L->cfg.N, L->cfg.K, L->cfg.K, false);
  return gp;
}

void add_dW(qe_layer* L, uint32_t p, float* dst, int32_t accumulate, float* temp, std::vector<qe::Launch>& ls) {
  const uint32_t K = L->cfg.K, N = L->cfg.N;
  ls.push_back(qe::make_gemm(dW_gemm(L, p, dst, accumulate, temp), L->ctx->dev->num_sms));
  if (temp) {
    qe::AccumParams ap{};
    ap.dst = (float4*)dst;
    ap.src = (const float4*)temp;
    ap.nvec = (uint64_t)N * K / 4;
    ap.accumulate = accumulate;
    ls.push_back(qe::make_accumulate(ap));
  }
}


}  // namespace qe_impl
