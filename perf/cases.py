"""The workloads this library's speed is judged on: what a training program has it do, through its public entry points.

A case is one pass of one of these programs (its "kind"):

  step     a whole optimizer step of a pipeline stage through `StepPlan.run` (one call, graph or eager), then the stage's
           optimizer boundary.  Every microbatch's forward, input gradient and deferred weight gradient of every linear.
  actions  the same step issued action by action (`Layer.forward` / `backward_dI` / `backward_dW`), as a scheduler that
           receives its microbatches one after the other does.
  chain    directly chained linears with the FP8 hand-off (`forward_chain`, `backward_dI_chain`), the weight gradients of
           a microbatch through `backward_dW_multi`.
  host     the step action by action with activations and gradients in pinned host memory (`forward_host`,
           `backward_dI_host`); the copies are part of the pass.
  cast     one tensor through `qe_quantize`, alone (a weight or an activation prepared for another consumer).
  gemm     one FP8 GEMM through `qe_gemm_fp8_ex`, alone.

Sizes are those of the repository's configurations (`paper_2609_23536_b200.inputs.CONFIGS`) and of the sequence-256
layers the paper trains (hidden / FFN 2048 / 8192 and 4096 / 11008), or generic.  The ranges declared by `draw`: tokens
256 to 4096, features 256 to 16384, both any multiple of 128 (casts: of 64); 1 to 16 microbatches, 1 to 16 linears;
histories from 4 to 1024 entries; margins 0 and 1; eager and graph execution; weight gradients on the execution stream or
overlapped on a second one; every output kind, operand format and operand major of the GEMM.
"""
import math

import torch

from paper_2609_23536_b200 import binding as qe
from paper_2609_23536_b200.schedules import peak_live, sched

DEVICE = "cuda:0"
GRAD_STD = 1e-3  # upstream gradients ~ N(0, 1e-3^2), activations ~ N(0, 1), weights ~ N(0, 0.02^2)


def _linears(text):
    """"2048x6144 2048x2048*3" -> [(K, N), ...] in the order the forward pass visits them."""
    out = []
    for word in text.split():
        shape, _, times = word.partition("*")
        k, n = shape.split("x")
        out += [(int(k), int(n))] * int(times or 1)
    return out


def listed():
    return [
        # The smallest step the layer takes (1F1B, no deferral, history of 4): twelve calls on tiny tensors, where nothing
        # but the calls' own cost counts.
        dict(name="linear_256", kind="actions", T=256, linears="256x256", M=4, H=4, margin=0, warmup=1, defer=0,
             graph=False, overlap=False, heavy_tail=False),
        # The paper's small model: one sequence of 256 tokens per microbatch through a 2048 / 8192 layer, issued action by
        # action from captured graphs, weight gradients overlapped on the second stream.
        dict(name="layer_2048_seq256", kind="actions", T=256, linears="2048x6144 2048x2048 2048x8192 8192x2048", M=4, H=16,
             margin=0, warmup=3, defer=3, graph=True, overlap=True, heavy_tail=False),
        # The paper's larger model: 256 tokens through a 4096 / 11008 layer, eight microbatches, one call per step.  Few
        # tokens against large weights: memory traffic of the gradients, few tiles per forward.
        dict(name="layer_4096_seq256", kind="step", T=256, linears="4096x12288 4096x4096 4096x11008 11008x4096", M=8, H=16,
             margin=0, warmup=3, defer=3, graph=True, overlap=False, heavy_tail=False),
        # A Llama-style block of hidden size 2048 at 2048 tokens, zero-bubble order, long history: the ordinary step.
        dict(name="block_2048", kind="step", T=2048, linears="2048x6144 2048x2048 2048x11264 5632x2048", M=8, H=1024,
             margin=0, warmup=3, defer=3, graph=True, overlap=False, heavy_tail=False),
        # A block of hidden size 4096 with 4096 tokens per microbatch: the largest GEMMs, bound by the tensor cores and the
        # power limit.
        dict(name="block_4096", kind="step", T=4096, linears="4096x6144 4096x4096 4096x28672 14336x4096", M=8, H=1024,
             margin=0, warmup=3, defer=3, graph=True, overlap=False, heavy_tail=False),
        # One square linear fed heavy-tailed activations with a margin (scale rollover), action by action in graph mode.
        dict(name="linear_4096_heavy_tail", kind="actions", T=4096, linears="4096x4096", M=8, H=16, margin=1, warmup=1,
             defer=2, graph=True, overlap=False, heavy_tail=True),
        # Many small linears of a stage and many microbatches: bound by the launches between which the work is cut.
        dict(name="small_linears_48", kind="step", T=512, linears="1024x1024*48", M=32, H=16, margin=0, warmup=3, defer=3,
             graph=True, overlap=False, heavy_tail=False),
        # Sizes that are odd multiples of 128 everywhere (a sequence trimmed to 1920 tokens, features off the powers of
        # two), eager, action by action.
        dict(name="block_ragged", kind="actions", T=1920, linears="2176x6528 2176x2176 2176x5760 5760x2176", M=4, H=64,
             margin=0, warmup=2, defer=1, graph=False, overlap=False, heavy_tail=False),
        # Sixteen linears that feed one another directly, FP8 all the way.
        dict(name="chain_1024", kind="chain", T=512, linears="1024x1024*16", M=8, H=16, margin=0, warmup=2, defer=2,
             graph=True, overlap=False, heavy_tail=False),
        # Activations and gradients that live in pinned host memory.
        dict(name="block_1024_host", kind="host", T=1024, linears="1024x3072 1024x1024 1024x5632 2816x1024", M=4, H=16,
             margin=0, warmup=2, defer=1, graph=True, overlap=False, heavy_tail=False),
        # One large tensor cast for another consumer, with its transposed copy and its maximum.
        dict(name="cast_transpose_4096x14336", kind="cast", rows=4096, cols=14336, e5m2=False, transposed=True, amax=True),
        # One GEMM of few rows against a square weight: fewer tiles than the chip has SMs.
        dict(name="gemm_512x4096x4096", kind="gemm", rows=512, cols=4096, contraction=4096, a_e5m2=False, a_mn=False,
             b_mn=False, out=0),
    ]


def draw(rng):
    # The same programs over the whole of their ranges: sizes spread over their logarithm, one in three of them an odd
    # multiple of the granule.
    def size(lo, hi, granule=128):
        v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        if rng.random() < 1 / 3:
            g = (int(v / granule) | 1) * granule
        else:
            g = round(v / (2 * granule)) * 2 * granule
        return min(max(g, lo), hi)

    def linears(h, most):
        shape = rng.choice(["block", "square", "mixed"])
        if shape == "block":
            ffn = size(h, min(2 * h + 2 * h // 3, 8192))
            return "%dx%d %dx%d %dx%d %dx%d" % (h, size(h, 3 * h), h, h, h, 2 * ffn, ffn, h)
        if shape == "square":
            return "%dx%d*%d" % (h, h, rng.randint(1, most))
        return " ".join("%dx%d" % (size(256, h), size(256, 2 * h)) for _ in range(rng.randint(1, most)))

    kind = rng.choice(["step", "step", "step", "actions", "actions", "actions", "chain", "host", "cast", "gemm"])
    if kind == "cast":
        return dict(kind=kind, rows=size(256, 16384, 64), cols=size(256, 16384, 64), e5m2=rng.random() < 0.5,
                    transposed=rng.random() < 0.5, amax=True)
    if kind == "gemm":
        rows = size(128, 8192)
        mn = rows % 256 == 0  # operands stored the other way round need an even number of 128-row tiles
        return dict(kind=kind, rows=rows, cols=size(256, 16384), contraction=size(256, 8192), a_e5m2=rng.random() < 0.5,
                    a_mn=mn and rng.random() < 0.3, b_mn=mn and rng.random() < 0.5, out=rng.choice([0, 0, 1, 2]))
    while True:
        T, h = size(256, 4096), size(256, 4096)
        case = dict(kind=kind, T=T, linears=linears(h, 8), M=rng.randint(2, 12), H=rng.choice([4, 16, 64, 1024]),
                    margin=rng.randint(0, 1), warmup=rng.randint(1, 3), defer=rng.randint(0, 3), graph=rng.random() < 0.6,
                    overlap=kind == "actions" and rng.random() < 0.4, heavy_tail=kind == "actions" and rng.random() < 0.2)
        if kind == "chain":  # the hand-off takes even numbers of 128-tiles
            h = max(256, h // 256 * 256)
            case.update(T=max(256, T // 256 * 256), linears="%dx%d*%d" % (h, h, rng.randint(2, 16)))
        w = work(case)
        if w["flops"] < 4e12 and w["bytes"] < (4e8 if kind == "host" else 6e9):
            return case


# --------------------------------------------------------------------------------------------------------------- inputs
def _normal(shape, std, g):
    return torch.randn(shape, generator=g, dtype=torch.float32, device=DEVICE).mul_(std).to(torch.bfloat16)


def _activations(shape, g, heavy_tail):
    if not heavy_tail:
        return _normal(shape, 1.0, g)
    # Student-t with 3 degrees of freedom, one element in a thousand a thousand times larger
    chi2 = sum(torch.randn(shape, generator=g, device=DEVICE).square_() for _ in range(3))
    x = torch.randn(shape, generator=g, device=DEVICE).div_(chi2.div_(3.0).sqrt_())
    spike = torch.rand(shape, generator=g, device=DEVICE) < 1e-3
    return torch.where(spike, x * 1000.0, x).to(torch.bfloat16)


class _Stage:
    """The linears of a stage with their inputs, outputs and gradient buffer."""

    def __init__(self, case, seed):
        g = torch.Generator(device=DEVICE)
        g.manual_seed(seed)
        self.case, self.kind = case, case["kind"]
        self.M = M = case["M"]
        T = case["T"]
        host = self.kind == "host"
        self.shapes = _linears(case["linears"])
        self.order = sched(M, case["warmup"], case["defer"])
        slots = peak_live(self.order)
        self.ctx = qe.Context(qe.GRAPH if case["graph"] else qe.EAGER, overlap_dw=case["overlap"],
                              step_window=max(2, case["warmup"] + case["defer"]))
        self.layers, self.offsets, at = [], [], 0
        for u, (K, N) in enumerate(self.shapes):
            self.layers.append(qe.Layer(self.ctx, T, K, N, case["H"], case["margin"], slots, _normal((N, K), 0.02, g), unit=u,
                                        host_io=host))
            self.offsets.append(at)
            at += N * K
        self.grad = torch.zeros(at, dtype=torch.float32, device=DEVICE)
        # one tensor per feature count, [linears with it, M, T, features]
        chain = self.kind == "chain"
        self.outputs = []
        self.X, x_all = self._tensors([K for K, _ in self.shapes][:1 if chain else None], host)
        self.dY, dy_all = self._tensors([N for _, N in self.shapes][-1:] if chain else [N for _, N in self.shapes], host)
        self.Y, y_all = self._tensors([N for _, N in self.shapes][-1:] if chain else [N for _, N in self.shapes], host)
        self.dX, dx_all = self._tensors([K for K, _ in self.shapes][:1 if chain else None], host)
        for t in x_all:
            for part in t.view(-1, T, t.shape[-1]):
                part.copy_(_activations(part.shape, g, case["heavy_tail"]))
        for t in dy_all:
            for part in t.view(-1, T, t.shape[-1]):
                part.copy_(_normal(part.shape, GRAD_STD, g))
        self.outputs = {"Y": y_all, "dX": dx_all, "grad": self.grad}
        self.epoch = 0
        self.plan = None
        if self.kind == "step":
            n = len(self.layers)
            acts = [(a, i, m) for a, m in self.order for i in (range(n) if a == "F" else range(n - 1, -1, -1))]
            self.plan = qe.StepPlan(self.ctx, self.layers, acts, M, self.X, self.Y, self.dY, self.dX, self.grad, self.offsets)

    def _tensors(self, features, host):
        """Per microbatch a list of [T, features[i]] views, and the tensors they are views of."""
        T, M = self.case["T"], self.M
        by = {f: torch.zeros((features.count(f), M, T, f), dtype=torch.bfloat16, device="cpu" if host else DEVICE, pin_memory=host)
              for f in dict.fromkeys(features)}
        at = [features[:i].count(f) for i, f in enumerate(features)]
        return [[by[f][at[i], m] for i, f in enumerate(features)] for m in range(M)], list(by.values())


def prepare(case, seed):
    if case["kind"] == "cast":
        g = torch.Generator(device=DEVICE)
        g.manual_seed(seed)
        rows, cols = case["rows"], case["cols"]
        x = _normal((rows, cols), GRAD_STD if case["e5m2"] else 1.0, g)
        return dict(case=case, x=x, scale=(57344.0 if case["e5m2"] else 448.0) / x.float().abs().max().reshape(1),
                    q=torch.zeros((rows, cols), dtype=torch.uint8, device=DEVICE),
                    qT=torch.zeros((cols, rows), dtype=torch.uint8, device=DEVICE) if case["transposed"] else None,
                    amax=torch.zeros(1, dtype=torch.float32, device=DEVICE))
    if case["kind"] == "gemm":
        g = torch.Generator(device=DEVICE)
        g.manual_seed(seed)
        M, N, Kc = case["rows"], case["cols"], case["contraction"]

        def fp8(shape, e5m2):
            x = torch.randn(shape, generator=g, dtype=torch.float32, device=DEVICE)
            top = 57344.0 if e5m2 else 448.0
            return (x * (top / x.abs().max())).to(torch.float8_e5m2 if e5m2 else torch.float8_e4m3fn).view(torch.uint8)

        alpha = lambda e5m2: torch.full((1,), 5.0 / (57344.0 if e5m2 else 448.0), dtype=torch.float32, device=DEVICE)  # noqa: E731
        return dict(case=case, a=fp8((Kc, M) if case["a_mn"] else (M, Kc), case["a_e5m2"]),
                    b=fp8((Kc, N) if case["b_mn"] else (N, Kc), False), alpha_a=alpha(case["a_e5m2"]), alpha_b=alpha(False),
                    d=torch.zeros((M, N), dtype=torch.float32 if case["out"] else torch.bfloat16, device=DEVICE),
                    amax=torch.zeros(1, dtype=torch.float32, device=DEVICE),
                    status=torch.zeros(1, dtype=torch.int32, device=DEVICE))
    return _Stage(case, seed)


# ------------------------------------------------------------------------------------------------------------- one pass
def _run_actions(s):
    tapes = {}
    n = len(s.layers)
    host = s.kind == "host"
    for a, m in s.order:
        for i in (range(n) if a == "F" else range(n - 1, -1, -1)):
            L = s.layers[i]
            if a == "F":
                tapes[m, i] = (L.forward_host if host else L.forward)(m, s.epoch, s.X[m][i], s.Y[m][i])
            elif a == "dI":
                (L.backward_dI_host if host else L.backward_dI)(tapes[m, i], s.dY[m][i], s.dX[m][i])
            else:
                L.backward_dW(tapes[m, i], s.grad, s.offsets[i])


def _run_chain(s):
    tapes = {}
    for a, m in s.order:
        if a == "F":
            tapes[m] = qe.forward_chain(s.layers, m, s.epoch, s.X[m][0], s.Y[m][0])
        elif a == "dI":
            qe.backward_dI_chain(s.layers, tapes[m], s.dY[m][0], s.dX[m][0])
        else:
            qe.backward_dW_multi(s.layers, tapes[m], s.grad, s.offsets)


def run(state):
    if isinstance(state, dict) and state["case"]["kind"] == "cast":
        if state["case"]["amax"]:
            state["amax"].zero_()  # the call takes the maximum with what is there
        qe.qe_quantize(state["x"], state["scale"], int(state["case"]["e5m2"]), state["q"], state["qT"],
                       state["amax"] if state["case"]["amax"] else None)
        return {"q": state["q"], "qT": state["qT"], "amax": state["amax"]}
    if isinstance(state, dict):
        c = state["case"]
        bf16 = c["out"] == 0
        if bf16:
            state["amax"].zero_()
        qe.qe_gemm_fp8_ex(state["a"], int(c["a_e5m2"]), c["a_mn"], state["b"], 0, c["b_mn"], state["alpha_a"], state["alpha_b"],
                          state["d"], c["out"], state["amax"] if bf16 else None, state["status"])
        return {"d": state["d"], "amax": state["amax"]} if bf16 else {"d": state["d"]}
    if state.plan is not None:
        state.plan.run()
    elif state.kind == "chain":
        _run_chain(state)
    else:
        _run_actions(state)
    qe.optimizer_boundary_all(state.layers, state.M)
    state.epoch += 1
    return state.outputs


# ----------------------------------------------------------------------------------------------------- work, tolerances
def work(case):
    if case["kind"] == "cast":
        n = case["rows"] * case["cols"]
        return {"bytes": (4 if case["transposed"] else 3) * n, "flops": 0}
    if case["kind"] == "gemm":
        M, N, Kc = case["rows"], case["cols"], case["contraction"]
        return {"bytes": (M + N) * Kc + M * N * (2 if case["out"] == 0 else 4), "flops": 2 * M * N * Kc}
    T, M, shapes = case["T"], case["M"], _linears(case["linears"])
    weights = sum(K * N for K, N in shapes)
    # X, dY in and Y, dX out in bf16 (a chain: at its two ends only), W in once, the gradient out once in FP32
    ends = shapes if case["kind"] != "chain" else [(shapes[0][0], shapes[-1][1])]
    return {"bytes": 4 * T * M * sum(K + N for K, N in ends) + 6 * weights, "flops": 6 * T * M * weights}


def tolerance(case):
    # Measured by running every listed case twice with tokens and features permuted (the same sums in another order): bf16
    # outputs differ by at most 7.6e-5 in norm and by one unit in the last place (2^-7 of the value at most), FP32 ones by
    # 2.3e-7 and 5.1e-6.  Stated: four times the former; for FP32 outputs alone what 32-bit sums of 16384 terms give.
    if case["kind"] == "cast":
        return "exact"
    if case["kind"] == "chain":
        # One rounding of the largest output of a linear moves the next linear's scale by one part in 256 and, with it,
        # three codes in a hundred by one step: 1.1e-2 (Y), 1.4e-2 (dX), 9e-3 (gradients), single elements 0.74.
        return {"rel": 0.03, "max": 0.99}
    if case["kind"] == "gemm" and case["out"]:
        return {"rel": 1e-5}
    return {"rel": 3e-4, "max": 0.032}
