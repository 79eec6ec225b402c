"""The library's host code linked with the CUDA runtime of tests/fake_runtime.cpp: what it enqueues on which stream, and in
which order, without a GPU."""
from __future__ import annotations

import ctypes as C
import os
import subprocess
from concurrent.futures import ThreadPoolExecutor

from paper_2609_23536_b200 import build

build.build()  # (the binding below takes its types and signatures from the module that loads the built library)
from paper_2609_23536_b200 import binding as qe  # noqa: E402

HERE = os.path.dirname(os.path.abspath(__file__))
HOST_SOURCES = ["error.cpp", "contract.cpp", "layer_core.cu", "layer.cu", "layer_group.cu", "standalone.cu", "noalloc.cu"]
CALLER = 7  # a caller's stream


def build_library(out_dir):
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    flags = ["-std=c++17", "-O1", "-g", "-fPIC", "-I", cuda, "-I", build.INCLUDE, "-I", build.CSRC]

    def compile_one(src):
        obj = os.path.join(out_dir, os.path.basename(src) + ".o")
        subprocess.run(["g++", "-x", "c++", *flags, "-c", src, "-o", obj], check=True)
        return obj

    with ThreadPoolExecutor(8) as pool:
        objs = list(pool.map(compile_one, [os.path.join(build.CSRC, s) for s in HOST_SOURCES] + [os.path.join(HERE, "fake_runtime.cpp")]))
    so = os.path.join(out_dir, "libqe_host.so")
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-o", so, *objs], check=True)
    return so


def load(so):
    lib = C.CDLL(so)
    for name, (res, args) in qe._SIGNATURES.items():
        fn = getattr(lib, name)
        fn.restype, fn.argtypes = res, args
    lib.fake_log.restype = lib.fake_replayed.restype = C.c_char_p
    lib.fake_fail.argtypes = [C.c_char_p, C.c_long]
    lib.fake_fail_alloc.argtypes = [C.c_long]
    lib.fake_pageable.argtypes = [C.c_size_t, C.c_size_t]
    lib.fake_alloc_left.restype = lib.fake_encodes.restype = C.c_long
    lib.fake_reset()
    return lib


class Stage:
    """Layers on one context, every buffer in host memory."""

    def __init__(self, lib, shapes, T=256, M=2, slots=2, mode=0, window=4, flags=0, host_io=False, exec_stream=None):
        self.lib, self.M, self.T, self.shapes = lib, M, T, shapes
        self.ctx, self.keep, self.layers, self.weights = C.c_void_p(), [], [], []
        cfg = qe.qe_ctx_config(exec_mode=mode, device=0, exec_stream=exec_stream, flags=flags, step_window=window)
        assert lib.qe_ctx_create(C.byref(cfg), C.byref(self.ctx)) == 0
        for u, (K, N) in enumerate(shapes):
            self.weights.append(self.buffer(2 * N * K))
            lc = qe.qe_layer_config(T=T, K=K, N=N, history_len=4, margin=0, slots=slots, unit=u, host_io=int(host_io),
                                    weight_dev=self.weights[-1])
            need = C.c_uint64()
            assert lib.qe_layer_workspace_bytes(C.byref(lc), C.byref(need)) == 0
            h = C.c_void_p()
            assert lib.qe_layer_create(self.ctx, C.byref(lc), self.buffer(need.value), need.value, C.byref(h)) == 0
            self.layers.append(h)
        self.elems = sum(K * N for K, N in shapes)
        self.grad = self.buffer(4 * self.elems)
        self.offsets = [sum(K * N for K, N in shapes[:i]) for i in range(len(shapes))]

    def buffer(self, nbytes):
        b = (C.c_char * (nbytes + 512))()
        self.keep.append(b)
        return (C.addressof(b) + 255) // 256 * 256

    def step(self, actions, layers=None, stream=CALLER, apart=False):
        """qe_step_run over (kind, layer index, microbatch) triples; the status.  apart: every unit has tensors of its own (a
        function of the layer and the microbatch: which buffers it has); otherwise a layer's outputs are its inputs."""
        idx = list(range(len(self.layers))) if layers is None else layers
        n = len(idx)
        hs = (C.c_void_p * n)(*[self.layers[i].value for i in idx])
        acts = (qe.qe_step_action * len(actions))(*[qe.qe_step_action(qe.ACT[k], l, m, 0) for k, l, m in actions])
        io = (qe.qe_step_io * (n * self.M))()
        for l, i in enumerate(idx):
            K, N = self.shapes[i]
            x, y = self.buffer(2 * self.T * K), self.buffer(2 * self.T * N)
            for m in range(self.M):
                io[l * self.M + m] = qe.qe_step_io(*(apart(l, m) if apart else (x, y, y, x)))
        offs = (C.c_uint64 * n)(*[self.offsets[i] for i in idx])
        return self.lib.qe_step_run(self.ctx, hs, n, acts, len(actions), self.M, io, self.grad, self.elems, offs, None, stream)

    def error(self):
        return self.lib.qe_last_error().decode()

    def close(self):
        for h in self.layers:
            self.lib.qe_layer_destroy(h)
        self.lib.qe_ctx_destroy(self.ctx)


class Order:
    """Which of the logged operations is sure to come before which: every stream and event carries, per stream, how many of
    that stream's operations precede it."""

    def __init__(self, log):
        self.ops, streams, events = [], {}, {}  # op: (kind, stream, words, what precedes it)
        for line in log.splitlines():
            kind, *w = line.split()
            if kind == "sync":
                continue
            if kind == "record":
                events[w[0]] = dict(streams.get(w[1], {}))
            elif kind == "wait":
                at = streams.setdefault(w[1], {})
                for s, n in events.get(w[0], {}).items():
                    at[s] = max(at.get(s, 0), n)
            else:
                at = streams.setdefault(w[0], {})
                at[w[0]] = at.get(w[0], 0) + 1
                self.ops.append((kind, w[0], w[1:], dict(at)))
        self.streams = streams

    def before(self, a, b):
        """op a is sure to be complete when op b (a later one of the log) starts."""
        return b[3].get(a[1], 0) >= a[3][a[1]]

    def seen_by(self, stream, a):
        """work that the stream is given now comes after op a"""
        return self.streams.get(str(stream), {}).get(a[1], 0) >= a[3][a[1]]

    def of(self, kind):
        return [o for o in self.ops if o[0] == kind]
