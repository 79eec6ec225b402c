// Layer API, several actions per call: grouped weight gradients, chained linears with FP8 hand-off, independent
// actions in shared launches (pairs, qe_run_together) and the whole-step call with its round planner.
#include "layer_impl.h"

using namespace qe_impl;

// The GEMMs of a chain in one launch where that is offered and fits the device, else one by one, each as `alone` has it.
template <class F>
static void push_chain(qe_ctx* ctx, std::vector<qe::GemmDesc>& gemms, std::vector<qe::Launch>& ls, F alone) {
  qe::Launch l;
  if (gemms.size() > 1 && ctx->chained_fit && qe::make_gemm_group(gemms.data(), (uint32_t)gemms.size(), ctx->dev->num_sms, &l)) {
    ls.push_back(std::move(l));
    return;
  }
  for (uint32_t i = 0; i < gemms.size(); ++i) {
    gemms[i].chained = false;
    alone(i, gemms[i]);
    ls.push_back(qe::make_gemm(gemms[i], ctx->dev->num_sms));
  }
}

// Weights cast anew: `together` of them or more in one launch (sixteen of 1024 x 1024 28 us for 82), fewer one by one.
static void push_refresh(const std::vector<qe::QuantParams>& casts, size_t together, std::vector<qe::Launch>& ls) {
  if (casts.size() >= together) ls.push_back(qe::make_quantize_multi(casts.data(), (uint32_t)casts.size()));
  else for (const qe::QuantParams& c : casts) ls.push_back(qe::make_quantize(c));
}

extern "C" {

int32_t qe_backward_dW_multi(qe_layer* const* layers, const qe_tape* tapes, uint32_t n, float* grad, uint64_t elems,
                             const uint64_t* offsets, void* caller_stream) try {
  if (!layers || !tapes || !offsets || n == 0 || n > QE_MAX_MULTI_DW) return fail(QE_ERR_BAD_ARG, "null argument or bad count %u", n);
  qe_ctx* ctx = layers[0] ? layers[0]->ctx : nullptr;
  for (uint32_t i = 0; i < n; ++i) {
    if (!layers[i] || layers[i]->ctx != ctx) return fail(QE_ERR_BAD_ARG, "layer %u is null or belongs to another context", i);
    for (uint32_t j = 0; j < i; ++j)
      if (layers[j] == layers[i]) return fail(QE_ERR_BAD_ARG, "layer %u appears twice", i);
  }
  // check (every layer, before anything runs) -> run -> commit
  int32_t acc[QE_MAX_MULTI_DW];
  int32_t st;
  for (uint32_t i = 0; i < n; ++i) {
    const uint64_t slice = (uint64_t)layers[i]->cfg.N * layers[i]->cfg.K;
    if ((st = qe_contract_dW_check(layers[i]->contract, &tapes[i], (uint64_t)(uintptr_t)grad, elems, offsets[i], slice, &acc[i])) != QE_OK)
      return st;
  }
  cudaStream_t caller = (cudaStream_t)caller_stream;
  Handshake handshake(ctx, caller);
  cudaStream_t run_on = ctx->exec_stream;
  if (ctx->dw_stream) {
    run_on = ctx->dw_stream;
    QE_CUDA(cudaEventRecord(ctx->ev_dw_in, caller));
    QE_CUDA(cudaStreamWaitEvent(run_on, ctx->ev_dw_in, 0));
    for (uint32_t i = 0; i < n; ++i) QE_CUDA(cudaStreamWaitEvent(run_on, layers[i]->ev_di[tapes[i].ref.slot], 0));
    ctx->stats.handoffs += 1;
  } else if ((st = handshake.in()) != QE_OK) {
    return st;
  }
  std::vector<qe::Launch> ls;
  DWBatch dwb(n);
  Fnv h;
  h.mix("dWmulti", 8);
  for (uint32_t i = 0; i < n; ++i) {
    const uint32_t p = tapes[i].ref.slot;
    dwb.add(ctx, layers[i], dW_gemm(layers[i], p, grad + offsets[i], acc[i], nullptr), ls);
    h.mix(&layers[i], sizeof(qe_layer*));
    h.mix(&p, sizeof(p));
  }
  dwb.flush(ctx, ls);
  if (ctx->exec_mode == QE_EXEC_GRAPH) {
    ActionGraph* g = keyed_graph(ctx, h.key, ls.size());
    if (!g) return fail(QE_ERR_BAD_ARG, "out of host memory");
    st = run_action(ctx, g, ls, run_on);
  } else {
    for (const qe::Launch& l : ls)
      if ((st = launch_eager(ctx, l, run_on)) != QE_OK) break;
  }
  if (st != QE_OK) return st;
  if (ctx->dw_stream) {
    for (uint32_t i = 0; i < n; ++i) {
      const uint32_t p = tapes[i].ref.slot;
      QE_CUDA(cudaEventRecord(layers[i]->ev_dw[p], run_on));
      layers[i]->dw_pending[p] = true;
    }
  } else if ((st = handshake.out()) != QE_OK) {
    return st;
  }
  for (uint32_t i = 0; i < n; ++i) {
    const uint64_t slice = (uint64_t)layers[i]->cfg.N * layers[i]->cfg.K;
    if ((st = qe_contract_dW_commit(layers[i]->contract, &tapes[i], (uint64_t)(uintptr_t)grad, offsets[i], slice)) != QE_OK) return st;
  }
  return QE_OK;
} QE_NO_MEMORY

// ------------------------------------------------------------------------------------------------ chained linears
static int32_t check_chain(qe_layer* const* layers, uint32_t n) {
  if (!layers || n == 0 || n > QE_MAX_CHAIN) return fail(QE_ERR_BAD_ARG, "null argument or bad chain length %u", n);
  for (uint32_t i = 0; i < n; ++i) {
    if (!layers[i] || layers[i]->ctx != layers[0]->ctx) return fail(QE_ERR_BAD_ARG, "layer %u is null or belongs to another context", i);
    for (uint32_t j = 0; j < i; ++j)
      if (layers[j] == layers[i]) return fail(QE_ERR_BAD_ARG, "layer %u appears twice", i);
    if (i && (layers[i]->cfg.T != layers[0]->cfg.T || layers[i]->cfg.K != layers[i - 1]->cfg.N))
      return fail(QE_ERR_SHAPE, "layer %u does not take layer %u's output ([%u, %u] after [%u, %u])", i, i - 1, layers[i]->cfg.T,
                  layers[i]->cfg.K, layers[i - 1]->cfg.T, layers[i - 1]->cfg.N);
  }
  // (whole 256-row tiles only, as for the shared launches)
  for (uint32_t i = 0; n > 1 && i < n; ++i)
    if (!qe::whole_row_tiles(layers[i]->cfg.N)) return fail(QE_ERR_UNSUPPORTED, "layer %u: N must be a multiple of 256 for the hand-off", i);
  return QE_OK;
}

int32_t qe_forward_chain(qe_layer* const* layers, uint32_t n, uint32_t mb, uint64_t gen, const void* x, void* y,
                         void* caller_stream, qe_tape* tapes_out) try {
  int32_t st = check_chain(layers, n);
  if (st != QE_OK) return st;
  if (!x || !y || !tapes_out) return fail(QE_ERR_BAD_ARG, "null argument");
  if (((uintptr_t)x | (uintptr_t)y) & 15u) return fail(QE_ERR_BAD_ARG, "x and y must be 16-byte aligned");
  int32_t refresh[QE_MAX_CHAIN];
  uint32_t p[QE_MAX_CHAIN];
  for (uint32_t i = 0; i < n; ++i)  // every layer's check before anything runs
    if ((st = qe_contract_forward_check(layers[i]->contract, mb, gen, &refresh[i], &p[i])) != QE_OK) return st;
  qe_ctx* ctx = layers[0]->ctx;
  cudaStream_t caller = (cudaStream_t)caller_stream;
  Handshake handshake(ctx, caller);
  if ((st = handshake.in()) != QE_OK) return st;
  std::vector<qe::Launch> ls;
  std::vector<qe::QuantParams> casts;  // of weights
  Fnv h;
  h.mix("Fchain", 7);
  for (uint32_t i = 0; i < n; ++i) {
    qe_layer* L = layers[i];
    if (L->dw_pending[p[i]]) {
      QE_CUDA(cudaStreamWaitEvent(ctx->exec_stream, L->ev_dw[p[i]], 0));
      L->dw_pending[p[i]] = false;
    }
    if (refresh[i]) casts.push_back(refresh_params(L));
    h.mix(&layers[i], sizeof(qe_layer*));
    h.mix(&p[i], sizeof(uint32_t));
    h.mix(&refresh[i], sizeof(int32_t));
  }
  std::vector<qe::GemmDesc> gemms(n);
  push_refresh(casts, qe::kLaunchChained, ls);
  for (uint32_t i = 0; i < n; ++i) {
    const bool last = i + 1 == n;
    add_forward(layers[i], p[i], i == 0 ? x : nullptr, last ? y : nullptr, ls, last ? nullptr : layers[i + 1], last ? 0 : p[i + 1], &gemms[i]);
    gemms[i].chained = n > 1;
  }
  push_chain(ctx, gemms, ls, [&](uint32_t i, qe::GemmDesc& g) {
    // A layer's Y is committed by the next layer's launch while that computes, the last layer's by its own tail: a tail with a
    // commit lengthens a launch by 2.8 us (ticket, dependent loads), of 8.4 for 512 x 1024 x 1024
    // (sixteen chained 1024 x 1024 linears 2016 -> 1721 us a step, twelve of 256 x 256 1395 -> 1194).
    if (i) g.before = commit_params(layers[i - 1], 1u << QE_CLASS_Y, 0, nullptr);
    if (i + 1 < n) g.commit.class_mask = 0;
  });
  if ((st = run_keyed(ctx, h.key, ls)) != QE_OK) return st;
  if ((st = handshake.out()) != QE_OK) return st;
  for (uint32_t i = 0; i < n; ++i)
    if ((st = qe_contract_forward_commit(layers[i]->contract, mb, &tapes_out[i])) != QE_OK) return st;
  return QE_OK;
} QE_NO_MEMORY

int32_t qe_backward_dI_chain(qe_layer* const* layers, const qe_tape* tapes, uint32_t n, const void* dy, void* dx,
                             void* caller_stream) try {
  int32_t st = check_chain(layers, n);
  if (st != QE_OK) return st;
  if (!tapes || !dy || !dx) return fail(QE_ERR_BAD_ARG, "null argument");
  if (((uintptr_t)dy | (uintptr_t)dx) & 15u) return fail(QE_ERR_BAD_ARG, "dy and dx must be 16-byte aligned");
  for (uint32_t i = 0; i < n; ++i)
    if ((st = qe_contract_dI_check(layers[i]->contract, &tapes[i])) != QE_OK) return st;
  qe_ctx* ctx = layers[0]->ctx;
  cudaStream_t caller = (cudaStream_t)caller_stream;
  Handshake handshake(ctx, caller);
  if ((st = handshake.in()) != QE_OK) return st;
  std::vector<qe::Launch> ls;
  Fnv h;
  h.mix("Bchain", 7);
  std::vector<qe::GemmDesc> gemms(n);
  for (uint32_t k = n; k-- > 0;) {  // last linear first
    const uint32_t pk = tapes[k].ref.slot;
    qe::GemmDesc& g = gemms[n - 1 - k];
    add_dI(layers[k], pk, k + 1 == n ? dy : nullptr, k == 0 ? dx : nullptr, ls, k ? layers[k - 1] : nullptr,
           k ? tapes[k - 1].ref.slot : 0, &g);
    g.chained = n > 1;
    h.mix(&layers[k], sizeof(qe_layer*));
    h.mix(&pk, sizeof(uint32_t));
  }
  push_chain(ctx, gemms, ls, [](uint32_t, qe::GemmDesc&) {});
  if ((st = run_keyed(ctx, h.key, ls)) != QE_OK) return st;
  if (ctx->dw_stream)
    for (uint32_t i = 0; i < n; ++i) QE_CUDA(cudaEventRecord(layers[i]->ev_di[tapes[i].ref.slot], ctx->exec_stream));
  if ((st = handshake.out()) != QE_OK) return st;
  for (uint32_t i = 0; i < n; ++i)
    if ((st = qe_contract_dI_commit(layers[i]->contract, &tapes[i])) != QE_OK) return st;
  return QE_OK;
} QE_NO_MEMORY

// ------------------------------------------------------------------------------------------------ F and dI together
// In the steady state of a split-backward schedule a stage holds a forward unit (microbatch m + k) and an input-
// gradient unit (microbatch m) at the same time.  Their chains through the layers are independent, so F of layer i
// and dI of layer j (two different layers) can share one GEMM launch: one fixed cost and common waves.
int32_t qe_forward_dI_pair(qe_layer* Lf, uint32_t mb, uint64_t gen, const void* x, void* y, qe_tape* tape_out,
                           qe_layer* Lb, const qe_tape* tape_b, const void* dy, void* dx, void* caller_stream) try {
  if (!Lf || !Lb || !x || !y || !tape_out || !tape_b || !dy || !dx) return fail(QE_ERR_BAD_ARG, "null argument");
  if (Lf == Lb || Lf->ctx != Lb->ctx) return fail(QE_ERR_BAD_ARG, "the two layers must be different layers of one context");
  if (((uintptr_t)x | (uintptr_t)y | (uintptr_t)dy | (uintptr_t)dx) & 15u) return fail(QE_ERR_BAD_ARG, "tensors must be 16-byte aligned");
  int32_t refresh = 0;
  uint32_t p = 0;
  int32_t st = qe_contract_forward_check(Lf->contract, mb, gen, &refresh, &p);  // both checks before anything runs
  if (st != QE_OK) return st;
  if ((st = qe_contract_dI_check(Lb->contract, tape_b)) != QE_OK) return st;
  qe_ctx* ctx = Lf->ctx;
  cudaStream_t caller = (cudaStream_t)caller_stream;
  Handshake handshake(ctx, caller);
  const uint32_t pb = tape_b->ref.slot;
  if ((st = handshake.in()) != QE_OK) return st;
  if (Lf->dw_pending[p]) {
    QE_CUDA(cudaStreamWaitEvent(ctx->exec_stream, Lf->ev_dw[p], 0));
    Lf->dw_pending[p] = false;
  }
  std::vector<qe::Launch> ls;
  if (refresh) add_refresh(Lf, ls);
  qe::GemmDesc g[2];
  qe::QuantParams c[2];
  add_forward(Lf, p, x, y, ls, nullptr, 0, &g[0], &c[0]);  // hands the casts and the GEMMs back
  add_dI(Lb, pb, dy, dx, ls, nullptr, 0, &g[1], &c[1]);
  ls.push_back(qe::make_quantize_multi(c, 2));  // both casts in one launch
  qe::Launch shared;
  if (qe::whole_row_tiles(g[0].M) && qe::whole_row_tiles(g[1].M) && qe::make_gemm_group(g, 2, ctx->dev->num_sms, &shared)) {
    ls.push_back(shared);
    ctx->stats.paired_f_di += 1;
  } else {  // T is an odd multiple of 128: one after the other
    ls.push_back(qe::make_gemm(g[0], ctx->dev->num_sms));
    ls.push_back(qe::make_gemm(g[1], ctx->dev->num_sms));
  }
  Fnv h;
  h.mix("FdI", 4);
  h.mix(&Lf, sizeof(Lf));
  h.mix(&Lb, sizeof(Lb));
  h.mix(&p, sizeof(p));
  h.mix(&pb, sizeof(pb));
  h.mix(&refresh, sizeof(refresh));
  if ((st = run_keyed(ctx, h.key, ls)) != QE_OK) return st;
  if (ctx->dw_stream) QE_CUDA(cudaEventRecord(Lb->ev_di[pb], ctx->exec_stream));
  if ((st = handshake.out()) != QE_OK) return st;
  if ((st = qe_contract_forward_commit(Lf->contract, mb, tape_out)) != QE_OK) return st;
  return qe_contract_dI_commit(Lb->contract, tape_b);
} QE_NO_MEMORY

// ------------------------------------------------------------------------------------------------ independent actions
namespace {
// An action on its way to the device: what its contract check said.
struct Prepared : qe_action {
  int32_t refresh = 0, acc = 0;
  uint32_t slot = 0;
};

// argument rules and every action's contract check; nothing is changed
int32_t together_prepare(qe_ctx* ctx, Prepared* acts, uint32_t n, float* grad, uint64_t grad_elems, bool* any_dw) {
  if (!ctx || !acts || n == 0 || n > QE_MAX_TOGETHER) return fail(QE_ERR_BAD_ARG, "null argument or bad count %u", n);
  for (uint32_t i = 0; i < n; ++i) {
    const qe_action& a = acts[i];
    if (a.kind > QE_ACT_DW || !a.layer || a.layer->ctx != ctx || !a.tape) return fail(QE_ERR_BAD_ARG, "action %u: bad kind, layer or tape", i);
    if (a.kind != QE_ACT_DW && (!a.in_dev || !a.out_dev || (((uintptr_t)a.in_dev | (uintptr_t)a.out_dev) & 15u)))
      return fail(QE_ERR_BAD_ARG, "action %u: input / output null or misaligned", i);
    for (uint32_t j = 0; j < i; ++j)
      if (acts[j].layer == a.layer && acts[j].kind == a.kind) return fail(QE_ERR_BAD_ARG, "actions %u and %u: same kind on the same layer", j, i);
    *any_dw |= a.kind == QE_ACT_DW;
  }
  if (*any_dw && !grad) return fail(QE_ERR_BAD_ARG, "gradient buffer is null");
  for (uint32_t i = 0; i < n; ++i) {
    Prepared& a = acts[i];
    qe_layer* L = a.layer;
    int32_t st;
    if (a.kind == QE_ACT_F) {
      st = qe_contract_forward_check(L->contract, a.mb, a.gen, &a.refresh, &a.slot);
    } else if (a.kind == QE_ACT_DI) {
      st = qe_contract_dI_check(L->contract, a.tape);
      a.slot = a.tape->ref.slot;
    } else {
      st = qe_contract_dW_check(L->contract, a.tape, (uint64_t)(uintptr_t)grad, grad_elems, a.grad_offset, (uint64_t)L->cfg.N * L->cfg.K, &a.acc);
      a.slot = a.tape->ref.slot;
    }
    if (st != QE_OK) return st;
  }
  return QE_OK;
}

// The GEMMs gemms[0..n) in as few launches as hold them, each launch with about as many.
void push_gemms(qe_ctx* ctx, const qe::GemmDesc* gemms, uint32_t n, std::vector<qe::Launch>& ls) {
  const uint32_t most = qe::most_committing(ctx->dev->num_sms);
  for (uint32_t launches = (n + most - 1) / most, share; launches; --launches, gemms += share, n -= share) {
    share = (n + launches - 1) / launches;
    qe::Launch l;
    if (share >= 2 && qe::make_gemm_group(gemms, share, ctx->dev->num_sms, &l)) ls.push_back(std::move(l));
    else for (uint32_t i = 0; i < share; ++i) ls.push_back(qe::make_gemm(gemms[i], ctx->dev->num_sms));
  }
}

// the launches: the casts in one launch, then every GEMM of whole 256-row tiles in one launch; weight gradients of
// several microbatches of one layer (whole-step call only) become one GEMM that adds their products up
// (refresh != null: the weight casts are collected there instead of being queued; apart: a round of a list whose tensors are
// apart: half-filled last row tiles share launches too; early: its casts may overlap what is before them)
int32_t together_build(qe_ctx* ctx, const Prepared* acts, uint32_t n, float* grad, std::vector<qe::Launch>& ls, Fnv* h,
                       std::vector<qe::QuantParams>* refresh = nullptr, bool apart = false, const qe::Announce& early = {}) {
  // The order of the launches' problems is settled before they are built: F and dI first (others wait for them), the weight
  // gradients' tiles after theirs; the longest tiles first (their contraction length decides a tile's duration), so that a
  // launch's last, partial wave is made of short ones (weight gradients: contraction over the tokens of all products).
  struct Product { const Prepared* first; uint32_t n; };  // a weight gradient: its first microbatch's action, its products
  std::vector<const Prepared*> chain_of;
  std::vector<Product> dw_of;
  const auto dw_product = [&](const qe_layer* L) {
    return std::find_if(dw_of.begin(), dw_of.end(), [&](const Product& d) { return d.first->layer == L; });
  };
  chain_of.reserve(n);
  for (int pass = 0; pass < 2; ++pass)
    for (uint32_t i = 0; i < n; ++i) {
      const Prepared& a = acts[i];
      if ((a.kind == QE_ACT_DW) != (pass == 1)) continue;
      if (h) {
        h->mix(&a.kind, sizeof(a.kind));
        h->mix(&a.layer, sizeof(a.layer));
        h->mix(&a.slot, sizeof(uint32_t));
        h->mix(&a.refresh, sizeof(int32_t));
      }
      if (pass == 0) {
        chain_of.push_back(&a);
      } else {
        const auto sum = dw_product(a.layer);  // this layer's of an earlier microbatch takes this one in
        if (sum != dw_of.end()) sum->n += 1;
        else dw_of.push_back({&a, 1});
      }
    }
  const auto contraction = [](const Prepared* a) { return a->kind == QE_ACT_F ? a->layer->cfg.K : a->layer->cfg.N; };
  std::stable_sort(chain_of.begin(), chain_of.end(), [&](const Prepared* x, const Prepared* y) { return contraction(x) > contraction(y); });
  std::stable_sort(dw_of.begin(), dw_of.end(), [](const Product& x, const Product& y) { return x.first->layer->cfg.T * x.n > y.first->layer->cfg.T * y.n; });
  std::vector<qe::GemmDesc> gemms, singles;  // those that share launches; those that go out one by one: half-filled last row tiles
  std::vector<qe::QuantParams> casts(chain_of.size());
  gemms.reserve(chain_of.size() + dw_of.size());
  const auto place = [&](uint32_t M) -> qe::GemmDesc& {
    std::vector<qe::GemmDesc>& to = apart || qe::whole_row_tiles(M) ? gemms : singles;
    to.emplace_back();
    return to.back();
  };
  for (size_t i = 0; i < chain_of.size(); ++i) {
    const Prepared& a = *chain_of[i];
    qe_layer* L = a.layer;
    qe::GemmDesc& gp = place(L->cfg.T);
    if (a.kind == QE_ACT_F) {
      if (L->dw_pending[a.slot]) {
        QE_CUDA(cudaStreamWaitEvent(ctx->exec_stream, L->ev_dw[a.slot], 0));
        L->dw_pending[a.slot] = false;
      }
      if (a.refresh && refresh) refresh->push_back(refresh_params(L));
      else if (a.refresh) add_refresh(L, ls);
      add_forward(L, a.slot, a.in_dev, a.out_dev, ls, nullptr, 0, &gp, &casts[i]);
    } else {
      add_dI(L, a.slot, a.in_dev, a.out_dev, ls, nullptr, 0, &gp, &casts[i]);
    }
  }
  const uint32_t n_chain = (uint32_t)gemms.size();
  // (a launch in which one adds products up computes all its weight gradients as sums)
  const auto shares = [&](const Product& d) { return apart || qe::whole_row_tiles(d.first->layer->cfg.N); };
  const bool sums = std::any_of(dw_of.begin(), dw_of.end(), [&](const Product& d) { return d.n > 1 && shares(d); });
  for (const Product& d : dw_of) {
    qe::GemmDesc& gp = place(d.first->layer->cfg.N);
    gp = dW_gemm(d.first->layer, d.first->slot, grad + d.first->grad_offset, d.first->acc, nullptr, d.n > 1 || (sums && shares(d)));
    for (const Prepared* a = d.first + 1; gp.nseg < d.n; ++a)
      if (a->kind == QE_ACT_DW && a->layer == d.first->layer) gp.add_product(a->slot, a->slot);
  }
  const uint32_t n_gemms = (uint32_t)gemms.size();
  for (size_t i = 0; i < casts.size(); i += qe::kMaxCasts) {  // all casts of the call in one launch
    const uint32_t m = (uint32_t)std::min<size_t>(qe::kMaxCasts, casts.size() - i);
    ls.push_back(m > 1 || early.word ? qe::make_quantize_multi(&casts[i], m, early) : qe::make_quantize(casts[i]));
  }
  for (const qe::GemmDesc& gp : singles) ls.push_back(qe::make_gemm(gp, ctx->dev->num_sms));
  if (n_gemms >= 2) {
    ctx->stats.grouped_dw += n_gemms - n_chain;
    ctx->stats.paired_f_di += n_chain ? 1 : 0;
  }
  // one launch where it holds them all; else weight gradients, which add products up, have launches of their own
  const uint32_t together = n_gemms <= qe::most_committing(ctx->dev->num_sms) ? n_gemms : n_chain;
  push_gemms(ctx, gemms.data(), together, ls);
  push_gemms(ctx, gemms.data() + together, n_gemms - together, ls);
  return QE_OK;
}

// Forward commits first: a forward's tape slot was chosen by its check, on the state before the call, and the kernels
// used it; a weight-gradient commit of the same layer releases a slot and must not come in between.
int32_t together_commit(const Prepared* acts, uint32_t n, float* grad) {
  for (uint32_t kind = QE_ACT_F; kind <= QE_ACT_DW; ++kind) {
    for (uint32_t i = 0; i < n; ++i) {
      const Prepared& a = acts[i];
      if (a.kind != kind) continue;
      qe_layer* L = a.layer;
      int32_t st;
      if (a.kind == QE_ACT_F) {
        st = qe_contract_forward_commit(L->contract, a.mb, a.tape);
        if (st == QE_OK && a.tape->ref.slot != a.slot) return fail(QE_ERR_ORDER, "forward committed to slot %u, ran in slot %u", a.tape->ref.slot, a.slot);
      } else if (a.kind == QE_ACT_DI) {
        st = qe_contract_dI_commit(L->contract, a.tape);
      } else {
        st = qe_contract_dW_commit(L->contract, a.tape, (uint64_t)(uintptr_t)grad, a.grad_offset, (uint64_t)L->cfg.N * L->cfg.K);
      }
      if (st != QE_OK) return st;
    }
  }
  return QE_OK;
}
}  // namespace

// host != 0: the in / out pointers of the F and dI actions are HOST buffers, staged through the layers' fixed device
// buffers like qe_forward_host / qe_backward_dI_host do (uploads of all actions first, read-backs after the kernels).
static int32_t run_together_impl(qe_ctx* ctx, qe_action* acts, uint32_t n, float* grad, uint64_t grad_elems, void* caller_stream,
                                 int host) {
  if (!ctx || !acts || n == 0 || n > QE_MAX_TOGETHER) return fail(QE_ERR_BAD_ARG, "null argument or bad count %u", n);
  Prepared dev[QE_MAX_TOGETHER];
  for (uint32_t i = 0; i < n; ++i) {
    static_cast<qe_action&>(dev[i]) = acts[i];
    if (!host || acts[i].kind > QE_ACT_DI || !acts[i].layer) continue;
    qe_layer* L = acts[i].layer;
    if (!L->x_stage) return fail(QE_ERR_BAD_ARG, "action %u: layer was created without host_io", i);
    if (!acts[i].in_dev) return fail(QE_ERR_BAD_ARG, "action %u: host input is null", i);
    dev[i].in_dev = acts[i].kind == QE_ACT_F ? L->x_stage : L->dy_stage;
    dev[i].out_dev = acts[i].kind == QE_ACT_F ? L->y_stage : L->dx_stage;
  }
  bool any_dw = false;
  int32_t st = together_prepare(ctx, dev, n, grad, grad_elems, &any_dw);  // check (every action, before anything runs)
  if (st != QE_OK) return st;
  cudaStream_t caller = (cudaStream_t)caller_stream;
  Handshake handshake(ctx, caller);
  if ((st = handshake.in()) != QE_OK) return st;
  if (host)
    for (uint32_t i = 0; i < n; ++i) {
      if (acts[i].kind > QE_ACT_DI) continue;
      const qe_layer_config& c = acts[i].layer->cfg;
      const size_t bytes = 2ull * c.T * (acts[i].kind == QE_ACT_F ? c.K : c.N);
      if ((st = host_upload(ctx, const_cast<void*>(dev[i].in_dev), acts[i].in_dev, bytes, caller)) != QE_OK) return st;
    }
  if (any_dw && ctx->dw_stream) {  // weight gradients issued earlier on the second stream accumulate into the same buffer
    QE_CUDA(cudaEventRecord(ctx->ev_dw_in, ctx->dw_stream));
    QE_CUDA(cudaStreamWaitEvent(ctx->exec_stream, ctx->ev_dw_in, 0));
  }
  std::vector<qe::Launch> ls;
  Fnv h;
  h.mix("together", 9);
  if ((st = together_build(ctx, dev, n, grad, ls, &h)) != QE_OK) return st;
  if ((st = run_keyed(ctx, h.key, ls)) != QE_OK) return st;  // ... run ...
  if (host)
    for (uint32_t i = 0; i < n; ++i) {
      if (acts[i].kind > QE_ACT_DI) continue;
      const qe_layer_config& c = acts[i].layer->cfg;
      const size_t bytes = 2ull * c.T * (acts[i].kind == QE_ACT_F ? c.N : c.K);
      if ((st = host_download(ctx, acts[i].out_dev, dev[i].out_dev, bytes)) != QE_OK) return st;
    }
  if (ctx->dw_stream)
    for (uint32_t i = 0; i < n; ++i)
      if (acts[i].kind == QE_ACT_DI) QE_CUDA(cudaEventRecord(acts[i].layer->ev_di[dev[i].slot], ctx->exec_stream));
  if ((st = handshake.out()) != QE_OK) return st;
  return together_commit(dev, n, grad);  // ... commit (the tapes are written through the callers' pointers)
}

int32_t qe_run_together(qe_ctx* ctx, qe_action* acts, uint32_t n, float* grad, uint64_t grad_elems, void* caller_stream) try {
  return run_together_impl(ctx, acts, n, grad, grad_elems, caller_stream, 0);
} QE_NO_MEMORY

int32_t qe_run_together_host(qe_ctx* ctx, qe_action* acts, uint32_t n, float* grad, uint64_t grad_elems, void* caller_stream) try {
  return run_together_impl(ctx, acts, n, grad, grad_elems, caller_stream, 1);
} QE_NO_MEMORY

// ------------------------------------------------------------------------------------------------ whole-step call
namespace {
struct Bytes { uintptr_t lo, hi; };

// Whether nothing that the list's actions write -- outputs, gradient slices, workspaces -- overlaps anything else they read or
// write: then only a layer's own order binds them, and the layers of a unit need not wait for one another.  (A null pointer: no.)
bool tensors_apart(qe_layer* const* layers, uint32_t n_layers, const qe_step_action* actions, uint32_t n_actions, uint32_t M,
                   const qe_step_io* io, const float* grad, const uint64_t* offsets) {
  // runs of one kind of tensor in the order of the list: mostly ascending as they come
  std::vector<Bytes> run[5];  // x, dy (read), weights (read), y, dx and the rest (written)
  enum { kX, kDY, kY, kDX, kRest };
  for (uint32_t i = 0; i < n_actions; ++i) {
    const qe_step_action& a = actions[i];
    if (a.kind > QE_ACT_DW || a.layer >= n_layers || a.mb >= M) return false;
    if (a.kind == QE_ACT_DW) continue;
    const qe_layer_config& c = layers[a.layer]->cfg;
    const qe_step_io& b = io[(size_t)a.layer * M + a.mb];
    const uintptr_t tk = 2ull * c.T * c.K, tn = 2ull * c.T * c.N;
    const uintptr_t in = (uintptr_t)(a.kind == QE_ACT_F ? b.x_dev : b.dy_dev), out = (uintptr_t)(a.kind == QE_ACT_F ? b.y_dev : b.dx_dev);
    if (!in || !out) return false;
    run[a.kind == QE_ACT_F ? kX : kDY].push_back({in, in + (a.kind == QE_ACT_F ? tk : tn)});
    run[a.kind == QE_ACT_F ? kY : kDX].push_back({out, out + (a.kind == QE_ACT_F ? tn : tk)});
  }
  std::vector<Bytes> weights;
  for (uint32_t l = 0; l < n_layers; ++l) {
    const qe_layer* L = layers[l];
    const uintptr_t nk = (uintptr_t)L->cfg.N * L->cfg.K, w = (uintptr_t)L->cfg.weight_dev, g = (uintptr_t)(grad + offsets[l]);
    weights.push_back({w, w + 2 * nk});
    run[kRest].push_back({(uintptr_t)L->st, (uintptr_t)L->st + L->ws_bytes});
    if (grad) run[kRest].push_back({g, g + 4 * nk});
  }
  run[kX].insert(run[kX].end(), weights.begin(), weights.end());
  const auto less = [](const Bytes& a, const Bytes& b) { return a.lo < b.lo; };
  for (std::vector<Bytes>& r : run)
    if (!std::is_sorted(r.begin(), r.end(), less)) std::sort(r.begin(), r.end(), less);
  // sweep by address: what is written may not begin before all that came before it has ended, nor anything before all that
  // is written has
  size_t at[5] = {};
  uintptr_t read_to = 0, written_to = 0;
  for (;;) {
    int best = -1;
    for (int k = 0; k < 5; ++k)
      if (at[k] < run[k].size() && (best < 0 || run[k][at[k]].lo < run[best][at[best]].lo)) best = k;
    if (best < 0) return true;
    const Bytes& b = run[best][at[best]++];
    const bool write = best >= kY;
    if (b.lo < written_to || (write && b.lo < read_to)) return false;
    (write ? written_to : read_to) = std::max(write ? written_to : read_to, b.hi);
  }
}

// Actions of a round of a list whose tensors are apart: forwards and input gradients for two launches (us a step with 28 / 56 / 112:
// 48 linears of 1024 at 512 tokens 5310 / 5240 / 4640, at 256 993 / 905 / 863; 64 of 512 at 512 1000 / 848 / 882; steps of up to
// 32 linears the same).
constexpr uint32_t kApartGroup = 2 * qe::kMaxProblems;
}  // namespace

int32_t qe_step_run(qe_ctx* ctx, qe_layer* const* layers, uint32_t n_layers, const qe_step_action* actions,
                    uint32_t n_actions, uint32_t M, const qe_step_io* io, float* grad, uint64_t grad_elems,
                    const uint64_t* offsets, float* temp, void* caller_stream) try {
  if (!ctx || !layers || !actions || !io || !offsets) return fail(QE_ERR_BAD_ARG, "null argument");
  if (n_layers == 0 || n_actions == 0 || M == 0 || M > QE_MAX_MICROBATCHES) return fail(QE_ERR_BAD_ARG, "empty list or bad microbatch count");
  if (temp && ((uintptr_t)temp & 15u)) return fail(QE_ERR_BAD_ARG, "temp_dev must be 16-byte aligned");
  for (uint32_t l = 0; l < n_layers; ++l)
    if (!layers[l] || layers[l]->ctx != ctx) return fail(QE_ERR_BAD_ARG, "layer %u is null or belongs to another context", l);
  cudaStream_t caller = (cudaStream_t)caller_stream;
  Handshake handshake(ctx, caller);

  std::vector<qe_tape> tapes((size_t)n_layers * M);
  std::vector<uint8_t> have((size_t)n_layers * M, 0);
  std::vector<qe::Launch> ls;
  ls.reserve(2 * (size_t)n_actions + n_layers);
  int32_t st = QE_OK;
  uint32_t k = 0;

  // ---- issuing: all pieces of the list behind one handshake
  int32_t run_status = QE_OK;
  uint32_t pieces = 0;
  Fnv list_key;  // over the list's identity
  if (ctx->exec_mode == QE_EXEC_GRAPH) {
    list_key.mix(layers, sizeof(qe_layer*) * n_layers);
    list_key.mix(actions, sizeof(qe_step_action) * n_actions);
    list_key.mix(&M, sizeof(M));
  }
  auto run_piece = [&](const std::vector<qe::Launch>& piece, bool as_graph) -> int32_t {
    if (pieces++ == 0) {
      const int32_t hs = handshake.in();
      if (hs != QE_OK) return hs;
      if (ctx->dw_stream) {
        // weight-gradient work issued earlier through the overlapped per-action path must finish first: this list's
        // dW kernels run on the execution stream and accumulate into the same buffer
        QE_CUDA(cudaEventRecord(ctx->ev_dw_in, ctx->dw_stream));
        QE_CUDA(cudaStreamWaitEvent(ctx->exec_stream, ctx->ev_dw_in, 0));
      }
    }
    if (ctx->exec_mode == QE_EXEC_GRAPH && as_graph) {
      Fnv h = list_key;
      h.mix(&pieces, sizeof(pieces));
      ActionGraph* g = keyed_graph(ctx, h.key, piece.size());
      if (!g) return fail(QE_ERR_BAD_ARG, "out of host memory");
      return run_action(ctx, g, piece);
    }
    for (const qe::Launch& l : piece) {
      const int32_t ls_status = launch_eager(ctx, l, ctx->exec_stream);
      if (ls_status != QE_OK) return ls_status;
    }
    return QE_OK;
  };

  // ---- issue plan.  The list is read as units (runs of actions of one kind and microbatch over distinct layers: a
  // forward, input-gradient or weight-gradient unit of the stage).  Units a stage holds at the same time are
  // independent, so the list is cut into rounds of actions whose predecessors were issued in earlier rounds -- the
  // previous layer of the own unit (F and dI walk their layers in list order), the same layer of the previous unit of
  // the kind, F before dI before dW of a (layer, microbatch), a free tape slot -- looking `window` units ahead, and a
  // round goes out as qe_run_together would issue it.  If no such plan exists (an illegal list) the action-by-action
  // pass below runs instead and reports the failing action.
  // Weight gradients: qe_plan_step collects a layer's and lets one launch add them up, as far as a sum stays within 8192
  // tokens and holds three products.  Few tokens make the destination's traffic the cost of a weight gradient: eight
  // microbatches of 256 tokens through a 4096 / 11008 layer 2860 -> 1890 us a step.  Blocks of eight microbatches, sums against
  // launches one by one: four products at 2048 tokens, hidden 1024 705 us for 794, 2048 2180 for 2410, 4096 9320 for 10310;
  // three at 2688, hidden 4096 13310 for 13970.  Tiles that last several times as long leave more of the chip idle at the end of
  // a launch; with the casts between the launches sums of two did not make up for that (hidden 2048 at 3072 tokens 4178 for 4094,
  // at 3584 4777 for 4641; hidden 4096 at 2816 11150 for 11087), which is where the line was drawn.  With the casts beside the
  // launches they do where tensors are apart (two products, hidden 4096 at 2816 14000 for 14600, at 3584 17270 for 17890; hidden
  // 2048 3460 for 3430 and 4140 for 4530): the line lies lower than it could there.
  uint32_t T_max = 0;
  for (uint32_t l = 0; l < n_layers; ++l) T_max = std::max(T_max, layers[l]->cfg.T);
  // A layer that the list names by more than one index is planned without sums (a sum belongs to one index), and two of its
  // actions of a kind may not meet in a round: the round's launch would commit the layer's scales twice.
  std::vector<qe_layer*> by_address(layers, layers + n_layers);
  std::sort(by_address.begin(), by_address.end());
  const bool repeated = std::adjacent_find(by_address.begin(), by_address.end()) != by_address.end();
  const uint32_t fit = 8192u / T_max, max_sum = repeated || fit < 3 ? 1u : std::min(qe::kMaxSegments, fit);
  // Where the list's tensors are apart (qe_plan_step_apart), a round takes every layer that is ready, not one of each unit: a
  // unit of n layers is one round instead of n, and half-filled last row tiles share its launches (of the tiles' rows a
  // sixteenth at 1920 tokens, a quarter at 384; launches of their own cost more).  us a step, layers in turn / at once:
  // 48 linears of 1024 x 1024 at 512 tokens 13250 / 5340; six of 1536 x 1536 at 1152 tokens (odd) 889 / 351; eight of 2048 x
  // 2048 at 768 1316 / 871; a 4096 / 11008 layer at 256 1776 / 1619; blocks of hidden 1024 at 3072 970 / 853, 2048 at 2048
  // 2900 / 2795; hidden 4096 at 4096, which the power limit bounds, the same.  (Both sides with the casts between the GEMMs.)
  std::vector<std::vector<uint32_t>> rounds;  // indices into actions[]
  bool apart = false;
  if (!temp && ctx->step_window > 1) {
    std::vector<uint32_t> slots(n_layers), live(n_layers), round_of(n_actions);
    for (uint32_t l = 0; l < n_layers; ++l) {
      slots[l] = layers[l]->cfg.slots;
      live[l] = layers[l]->contract->live_tapes();
    }
    uint32_t n_rounds = 0;
    apart = !repeated && tensors_apart(layers, n_layers, actions, n_actions, M, io, grad, offsets) &&
            qe_plan_step_apart(actions, n_actions, n_layers, M, slots.data(), live.data(), ctx->step_window, kApartGroup, max_sum,
                               round_of.data(), &n_rounds) == QE_OK;
    if (apart || (max_sum > 1 && qe_plan_step(actions, n_actions, n_layers, M, slots.data(), live.data(), ctx->step_window,
                                     QE_MAX_TOGETHER, max_sum, round_of.data(), &n_rounds) == QE_OK) ||
        qe_plan_rounds(actions, n_actions, n_layers, M, slots.data(), live.data(), ctx->step_window, QE_MAX_TOGETHER,
                       round_of.data(), &n_rounds) == QE_OK) {
      rounds.resize(n_rounds);
      for (uint32_t i = 0; i < n_actions; ++i) rounds[round_of[i]].push_back(i);
    }
  }
  // Weights that are to be cast anew: the casts of a piece (below) go out together ahead of it instead of one by one between
  // the rounds of the warm-up.
  std::vector<qe::QuantParams> refresh;
  auto put_refresh = [&] {
    std::vector<qe::Launch> first;
    for (size_t i = 0; i < refresh.size(); i += qe::kMaxCasts) {
      const uint32_t n = (uint32_t)std::min<size_t>(qe::kMaxCasts, refresh.size() - i);
      first.push_back(n > 1 ? qe::make_quantize_multi(&refresh[i], n) : qe::make_quantize(refresh[i]));
    }
    ls.insert(ls.begin(), std::make_move_iterator(first.begin()), std::make_move_iterator(first.end()));
    refresh.clear();
  };
  uint32_t waiting = 0;  // actions in the piece that is being put together
  // Commits that GEMM launches announce to casts (Announce), and what their count has come to.  In graph mode the numbers are
  // the piece's own, the same at every replay, and its last launch sets the count back; in eager mode they go on.
  uint32_t* const commits = &layers[0]->st->commits;
  const bool by_graphs = ctx->exec_mode == QE_EXEC_GRAPH;
  uint32_t announced = by_graphs ? 0 : layers[0]->commits;
  auto end_of_piece = [&] {
    if (by_graphs && announced) qe::withdraw_commits(&ls.back(), commits);
    if (by_graphs) announced = 0;
    else layers[0]->commits = announced;
  };
  std::vector<uint64_t> freed(n_layers, 0), freed_before(n_layers, 0);  // slots that the weight gradients of a round release
  std::vector<Prepared> acts;
  for (size_t r = 0; r < rounds.size() && st == QE_OK; ++r) {
    // check -> commit per action (all F first: a slot that a dW of the round releases is not theirs to take), then the
    // launches of those that passed
    acts.clear();
    bool early = apart && !ls.empty() && !ctx->launch_failed, casts = false;
    freed_before.swap(freed);
    std::fill(freed.begin(), freed.end(), 0);
    for (size_t i = 0; repeated && i < rounds[r].size(); ++i)
      for (size_t j = 0; j < i; ++j) {
        const qe_step_action &a = actions[rounds[r][j]], &b = actions[rounds[r][i]];
        if (a.kind == b.kind && layers[a.layer] == layers[b.layer])
          st = fail(QE_ERR_BAD_ARG, "actions %u and %u: same kind on the same layer", rounds[r][j], rounds[r][i]);
      }
    if (st != QE_OK) k = rounds[r][0];
    for (uint32_t kind = QE_ACT_F; kind <= QE_ACT_DW && st == QE_OK; ++kind) {
      for (uint32_t gi : rounds[r]) {
        const qe_step_action& a = actions[gi];
        if (a.kind != kind) continue;
        const size_t u = (size_t)a.layer * M + a.mb;
        qe_layer* L = layers[a.layer];
        const uint64_t slice = (uint64_t)L->cfg.N * L->cfg.K;
        Prepared p;
        const void* in = a.kind == QE_ACT_F ? io[u].x_dev : io[u].dy_dev;
        void* out = a.kind == QE_ACT_F ? io[u].y_dev : io[u].dx_dev;
        if (a.kind == QE_ACT_DW) {
          st = !grad ? fail(QE_ERR_BAD_ARG, "gradient buffer is null")
                     : qe_contract_dW_check(L->contract, &tapes[u], (uint64_t)(uintptr_t)grad, grad_elems, offsets[a.layer], slice, &p.acc);
          p.slot = tapes[u].ref.slot;
          if (st == QE_OK) st = qe_contract_dW_commit(L->contract, &tapes[u], (uint64_t)(uintptr_t)grad, offsets[a.layer], slice);
          freed[a.layer] |= 1ull << (p.slot & 63u);
        } else if (!in || !out || (((uintptr_t)in | (uintptr_t)out) & 15u)) {
          st = fail(QE_ERR_BAD_ARG, "input / output null or misaligned");
        } else if (a.kind == QE_ACT_F) {
          st = qe_contract_forward_check(L->contract, a.mb, L->contract->e_W, &p.refresh, &p.slot);
          if (st == QE_OK) st = qe_contract_forward_commit(L->contract, a.mb, &tapes[u]);
          casts = true;
          early = early && !(freed_before[a.layer] >> (p.slot & 63u) & 1u);  // the GEMMs of the round before still read this slot
        } else {
          st = qe_contract_dI_check(L->contract, &tapes[u]);
          p.slot = tapes[u].ref.slot;
          if (st == QE_OK) st = qe_contract_dI_commit(L->contract, &tapes[u]);
          casts = true;
        }
        if (st != QE_OK) {
          k = gi;
          break;
        }
        static_cast<qe_action&>(p) = qe_action{a.kind, a.mb, 0, L, in, out, &tapes[u], offsets[a.layer]};
        acts.push_back(p);
      }
    }
    char why[512];  // (a build can only fail on a CUDA error, which then is the one to report)
    if (st != QE_OK) std::snprintf(why, sizeof(why), "%s", qe_last_error());
    qe::Announce before;  // (the launch at the end of the list is the GEMM launch that these casts come after)
    if (early && casts && !acts.empty()) before = {commits, announced += qe::announce_commits(&ls.back(), commits)};
    const int32_t built = acts.empty() ? QE_OK : together_build(ctx, acts.data(), (uint32_t)acts.size(), grad, ls, nullptr, &refresh, apart, before);
    if (st != QE_OK) st = fail(st, "%s", why);
    else if (built != QE_OK) {
      st = built;
      k = rounds[r][0];
    }
    // A long list goes out in pieces (in graph mode each a graph of its own), so that the device works on one while the host
    // prepares the next: a first one soon, the next while that one runs, later ones so long that the gaps between graphs do
    // not count.  us a step as one graph / in pieces of 96 / of 384 / of 96, 192 and then 384 actions: 48 linears of 1024, 32
    // microbatches of 512 tokens 5350 / 4685 / 4685 / 4670, eight of 256 1040 / 880 / 938 / 862; blocks, which are two or three
    // pieces, the same.
    waiting += (uint32_t)acts.size();
    if (st == QE_OK && waiting >= (pieces < 2 ? 96u << pieces : 384u) && r + 1 < rounds.size()) {
      end_of_piece();
      put_refresh();
      run_status = run_piece(ls, true);
      ls.clear();
      waiting = 0;
      if (run_status != QE_OK) break;
    }
  }
  end_of_piece();
  put_refresh();
  if (!rounds.empty()) k = st == QE_OK ? n_actions : k;

  // ---- host pass: check -> collect launches -> commit, action by action (Algorithm 1)
  DWBatch dwb(n_layers);
  for (; rounds.empty() && k < n_actions && st == QE_OK; ++k) {
    const qe_step_action& a = actions[k];
    if (a.kind != QE_ACT_DW) dwb.flush(ctx, ls);
    if (a.layer >= n_layers || a.mb >= M || a.kind > QE_ACT_DW) {
      st = fail(QE_ERR_BAD_ARG, "action %u: kind %u layer %u mb %u", k, a.kind, a.layer, a.mb);
      break;
    }
    qe_layer* L = layers[a.layer];
    const size_t u = (size_t)a.layer * M + a.mb;
    const qe_step_io& b = io[u];
    if (a.kind == QE_ACT_F) {
      int32_t refresh = 0;
      uint32_t p = 0;
      if (!b.x_dev || !b.y_dev || (((uintptr_t)b.x_dev | (uintptr_t)b.y_dev) & 15u)) { st = fail(QE_ERR_BAD_ARG, "action %u: x/y null or misaligned", k); break; }
      if ((st = qe_contract_forward_check(L->contract, a.mb, L->contract->e_W, &refresh, &p)) != QE_OK) break;
      if (L->dw_pending[p]) {  // a dW issued earlier through the overlapped per-action path still reads this slot
        cudaStreamWaitEvent(ctx->exec_stream, L->ev_dw[p], 0);
        L->dw_pending[p] = false;
      }
      if (refresh) add_refresh(L, ls);
      add_forward(L, p, b.x_dev, b.y_dev, ls);
      st = qe_contract_forward_commit(L->contract, a.mb, &tapes[u]);
      have[u] = 1;
    } else if (a.kind == QE_ACT_DI) {
      if (!have[u]) { st = fail(QE_ERR_ORDER, "action %u: dI before F in this list", k); break; }
      if (!b.dy_dev || !b.dx_dev || (((uintptr_t)b.dy_dev | (uintptr_t)b.dx_dev) & 15u)) { st = fail(QE_ERR_BAD_ARG, "action %u: dy/dx null or misaligned", k); break; }
      if ((st = qe_contract_dI_check(L->contract, &tapes[u])) != QE_OK) break;
      add_dI(L, tapes[u].ref.slot, b.dy_dev, b.dx_dev, ls);
      st = qe_contract_dI_commit(L->contract, &tapes[u]);
    } else {
      if (!have[u]) { st = fail(QE_ERR_ORDER, "action %u: dW before F in this list", k); break; }
      const uint64_t slice = (uint64_t)L->cfg.N * L->cfg.K;
      int32_t acc = 0;
      if ((st = qe_contract_dW_check(L->contract, &tapes[u], (uint64_t)(uintptr_t)grad, grad_elems, offsets[a.layer], slice, &acc)) != QE_OK) break;
      if (temp) add_dW(L, tapes[u].ref.slot, grad + offsets[a.layer], acc, temp, ls);
      else dwb.add(ctx, L, dW_gemm(L, tapes[u].ref.slot, grad + offsets[a.layer], acc, nullptr), ls);
      st = qe_contract_dW_commit(L->contract, &tapes[u], (uint64_t)(uintptr_t)grad, offsets[a.layer], slice);
    }
  }
  dwb.flush(ctx, ls);
  const int32_t check_status = st;
  char saved_msg[512];
  std::snprintf(saved_msg, sizeof(saved_msg), "%s", qe_last_error());

  // ---- device pass: the launches of every action that passed (in graph mode the ones that are not on their way yet)
  if (run_status == QE_OK && !ls.empty()) run_status = run_piece(ls, check_status == QE_OK);
  ctx->launch_failed |= run_status != QE_OK;
  if (run_status == QE_OK && pieces) run_status = handshake.out();
  if (check_status != QE_OK || run_status != QE_OK) {
    // failure boundary: outstanding tapes aborted, arenas unusable for the epoch
    for (uint32_t l = 0; l < n_layers; ++l) qe_contract_abort(layers[l]->contract);
    if (check_status != QE_OK) return fail(check_status, "step aborted at action %u: %s", k, saved_msg);
    return run_status;
  }
  return QE_OK;
} catch (const std::bad_alloc&) {  // (the layers were looked at before anything was allocated)
  for (uint32_t l = 0; l < n_layers; ++l) qe_contract_abort(layers[l]->contract);
  return qe::out_of_memory();
}

}  // extern "C"
