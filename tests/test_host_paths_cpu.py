"""What the layer API's host code enqueues, checks and refuses, on a CUDA runtime that only writes down what it is asked."""
import pytest

import fake_runtime


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    return fake_runtime.load(fake_runtime.build_library(str(tmp_path_factory.mktemp("host"))))


@pytest.fixture(autouse=True)
def clean(lib):
    lib.fake_reset()
    yield
    lib.fake_reset()


BAD_ARG, CUDA = -1, -16


def test_one_layer_under_two_indices_never_shares_a_launch_with_itself(lib):
    """Two actions of a kind on one layer in one launch would commit its scales twice, and two indices' weight gradients
    would be added up in one sum, beyond the products that a sum has room for."""
    s = fake_runtime.Stage(lib, [(256, 256)], M=16, slots=16, window=8)
    acts = [(k, m // 8, m) for k in ("F", "dI", "dW") for m in (0, 8, 1, 9, 2, 10, 3, 11, 4, 12, 5, 13, 6, 14, 7, 15)]
    assert s.step(acts, layers=[0, 0]) == BAD_ARG and "same layer" in s.error()
    assert b"launch" not in lib.fake_log()
    s.close()
    s = fake_runtime.Stage(lib, [(256, 256)], M=2, slots=2, window=1)  # action by action the list is a legal one
    assert s.step([("F", 0, 0), ("F", 1, 1), ("dI", 0, 0), ("dI", 1, 1), ("dW", 0, 0), ("dW", 1, 1)], layers=[0, 0]) == 0
    s.close()


def _actions(M, n):
    return [(k, l, m) for m in range(M) for k, order in (("F", range(n)), ("dI", range(n - 1, -1, -1)), ("dW", range(n - 1, -1, -1)))
            for l in order]


@pytest.mark.parametrize("mode,fn,nth", [(1, "cudaGraphInstantiate", 2), (1, "cudaGraphLaunch", 2), (1, "cudaStreamBeginCapture", 2),
                                         (0, "cudaLaunchKernelExC", 5), (0, "cudaLaunchKernelExC", 90)])
def test_a_step_that_fails_part_way_leaves_the_callers_stream_behind_what_is_running(lib, mode, fn, nth):
    s = fake_runtime.Stage(lib, [(256, 256)] * 20, M=4, slots=4, mode=mode, window=4)
    lib.fake_reset()
    lib.fake_fail(fn.encode(), nth)
    assert s.step(_actions(4, 20)) == CUDA
    order = fake_runtime.Order(lib.fake_log().decode())
    launches = order.of("launch")
    assert launches and all(order.seen_by(fake_runtime.CALLER, x) for x in launches)
    s.close()


def _calls(s, lib):
    """One after the other the calls that put work on the execution stream; the status of each."""
    import ctypes as C

    from paper_2609_23536_b200 import binding as qe

    T, (K, N) = s.T, s.shapes[0]
    x, y, grad, at = s.buffer(2 * T * K), s.buffer(2 * T * N), s.grad, fake_runtime.CALLER
    n = len(s.layers)
    hs, offs = (C.c_void_p * n)(*[h.value for h in s.layers]), (C.c_uint64 * n)(*s.offsets)
    tapes, t2 = (qe.qe_tape * n)(), (qe.qe_tape * n)()
    yield "qe_forward_chain", lambda: lib.qe_forward_chain(hs, n, 0, 0, x, y, at, tapes)
    yield "qe_backward_dI_chain", lambda: lib.qe_backward_dI_chain(hs, tapes, n, y, x, at)
    yield "qe_backward_dW_multi", lambda: lib.qe_backward_dW_multi(hs, tapes, n, grad, s.elems, offs, at)
    for i in range(n):
        yield "qe_forward", lambda: lib.qe_forward(hs[i], 1, 0, x, y, at, C.byref(t2[i]))
    acts = (qe.qe_action * 1)(qe.qe_action(1, 1, 0, hs[0], y, x, C.pointer(t2[0]), 0))
    yield "qe_run_together", lambda: lib.qe_run_together(s.ctx, acts, 1, grad, s.elems, at)
    yield "qe_backward_dI", lambda: lib.qe_backward_dI(hs[1], C.byref(t2[1]), y, x, at)
    temp = s.buffer(4 * N * K)
    yield "qe_backward_dW_staged", lambda: lib.qe_backward_dW_staged(hs[0], C.byref(t2[0]), grad, s.elems, offs[0], temp, at)
    yield "qe_backward_dW", lambda: lib.qe_backward_dW(hs[1], C.byref(t2[1]), grad, s.elems, offs[1], at)
    yield "qe_forward", lambda: lib.qe_forward(hs[0], 2, 0, x, y, at, C.byref(t2[0]))
    yield "qe_forward_dI_pair", lambda: lib.qe_forward_dI_pair(hs[1], 2, 0, x, y, C.byref(t2[1]), hs[0], C.byref(t2[0]), y, x, at)


def test_a_call_whose_last_launch_fails_leaves_the_callers_stream_behind_the_others(lib):
    shapes = [(256, 256)] * 3
    plain = fake_runtime.Stage(lib, shapes, slots=4)
    for i, (name, call) in enumerate(_calls(plain, lib)):
        lib.fake_reset()
        assert call() == 0, (name, plain.error())
        n = len(fake_runtime.Order(lib.fake_log().decode()).of("launch"))
        if n < 2:
            continue
        s = fake_runtime.Stage(lib, shapes, slots=4)
        for j, (_, other) in enumerate(_calls(s, lib)):
            if j == i:
                lib.fake_reset()
                lib.fake_fail(b"cudaLaunchKernelExC", n)
                assert other() == CUDA
                break
            assert other() == 0
        order = fake_runtime.Order(lib.fake_log().decode())
        assert len(order.of("launch")) == n - 1
        assert all(order.seen_by(fake_runtime.CALLER, x) for x in order.of("launch")), name
        s.close()
    plain.close()


@pytest.mark.parametrize("own_stream", [True, False], ids=["callers-stream", "execution-stream"])
def test_a_host_input_that_an_earlier_call_reads_back_is_uploaded_after_that(lib, own_stream):
    import ctypes as C

    from paper_2609_23536_b200 import binding as qe

    s = fake_runtime.Stage(lib, [(256, 256)] * 3, host_io=True, slots=4, exec_stream=None if own_stream else fake_runtime.CALLER)
    a, b, c, d = (s.buffer(2 * s.T * 256) for _ in range(4))
    tape = qe.qe_tape()

    def forward(layer, mb, x, y):
        assert lib.qe_forward_host(s.layers[layer], mb, 0, x, y, fake_runtime.CALLER, C.byref(tape)) == 0

    lib.fake_reset()
    forward(0, 0, a, b)
    forward(1, 0, b, c)                        # the whole buffer
    forward(2, 0, c + 2 * 256 * 255, a)        # its last row
    order = fake_runtime.Order(lib.fake_log().decode())
    up, down = order.of("h2d"), order.of("d2h")
    assert order.before(down[0], up[1]) and order.before(down[1], up[2])
    lib.fake_reset()
    forward(0, 1, a, b)
    forward(1, 1, d, c)                        # other memory: the link is used in both directions at once
    order = fake_runtime.Order(lib.fake_log().decode())
    assert order.before(order.of("d2h")[0], order.of("h2d")[1]) == own_stream
    lib.fake_reset()
    for i in range(600):                       # however many read-backs lie in between
        assert lib.qe_abort_step(s.layers[0]) == 0 and lib.qe_arena_rebuild(s.layers[0]) == 0
        forward(0, 0, a, b if i == 0 else d)
    forward(2, 1, b, c)
    order = fake_runtime.Order(lib.fake_log().decode())
    assert order.before(order.of("d2h")[0], order.of("h2d")[-1])
    s.close()


def test_the_call_that_must_not_allocate_takes_no_heap_memory(lib):
    import ctypes as C

    buf = (C.c_char * (1 << 20))()
    a = (C.addressof(buf) + 255) // 256 * 256
    call = lambda: lib.qe_gemm_fp8_staged_noalloc(a, 0, a, 0, 256, 256, 256, a, a, a, 0, a, None)  # noqa: E731
    assert call() == 0  # the warm-up, which may
    lib.fake_fail_alloc(1)
    assert call() == 0 and lib.fake_alloc_left() == 1


def out_of_memory(so):
    """(runs in a process of its own) Every allocation of every call fails in turn: the call says so, leaves the caller's
    stream behind what it issued and works when it is made again."""
    lib = fake_runtime.load(so)

    def attempts(call, again=None):
        nth = 0
        while True:
            nth += 1
            lib.fake_reset()
            lib.fake_fail_alloc(nth)
            st = call()
            if lib.fake_alloc_left() > 0:
                assert st == 0, (nth, st, lib.qe_last_error())
                lib.fake_reset()
                return nth
            # (a step that finds no memory for one issue plan may still run by another)
            assert st == BAD_ARG and b"out of host memory" in lib.qe_last_error() or (st == 0 and again), (st, lib.qe_last_error())
            order = fake_runtime.Order(lib.fake_log().decode())
            assert all(order.seen_by(fake_runtime.CALLER, x) for kind in ("launch", "h2d", "d2h") for x in order.of(kind))
            if again:
                again()

    import ctypes as C

    from paper_2609_23536_b200 import binding as qe

    for mode in (0, 1):
        s = fake_runtime.Stage(lib, [(256, 256)] * 3, T=384, slots=4, mode=mode)
        for name, call in _calls(s, lib):
            assert attempts(call) > 1, name
        for T, pieces in ((256, 1), (1024, 2), (2048, 4)):  # (nothing is on its way before all that the call needs is there)
            h = fake_runtime.Stage(lib, [(256, 2048)], T=T, host_io=True, slots=4, mode=mode)
            x, y, tape = h.buffer(2 * T * 256), h.buffer(2 * T * 2048), qe.qe_tape()
            assert attempts(lambda: lib.qe_forward_host(h.layers[0], 0, 0, x, y, fake_runtime.CALLER, C.byref(tape))) > 1
            assert attempts(lambda: lib.qe_backward_dI_host(h.layers[0], C.byref(tape), y, x, fake_runtime.CALLER)) > 1
            h.close()
        view, window = qe.qe_state_view(), (C.c_float * 16)()
        attempts(lambda: lib.qe_get_state(s.layers[0], C.byref(view), window, None))
        out = (C.c_char * 65536)()
        attempts(lambda: lib.qe_read_fp8(s.layers[0], 5, 0, out, 65536))
        s.close()
        s = fake_runtime.Stage(lib, [(256, 256)] * 12, M=4, slots=4, mode=mode)
        rebuild = lambda: [lib.qe_arena_rebuild(h) for h in s.layers]  # noqa: E731
        assert attempts(lambda: s.step(_actions(4, 12)), rebuild) > 100
        s.close()
    h, c, reg = C.c_void_p(), C.c_void_p(), C.c_void_p()
    attempts(lambda: lib.qe_registry_create(C.byref(reg)))
    attempts(lambda: lib.qe_contract_create(4, 0, 0, 0, reg, C.byref(c)))
    print("all attempts made")


def test_no_allocation_that_fails_ends_the_process(lib):
    import os
    import subprocess
    import sys

    here = os.path.dirname(os.path.abspath(__file__))
    code = "import sys; sys.path[:0] = sys.argv[2:]; import test_host_paths_cpu as t; t.out_of_memory(sys.argv[1])"
    r = subprocess.run([sys.executable, "-c", code, lib._name, here, os.path.dirname(here)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "all attempts made" in r.stdout, r.stderr[-2000:]


def test_standalone_gemms_encode_one_map_per_operand_and_output(lib):
    import ctypes as C

    from paper_2609_23536_b200 import binding as qe

    buf = (C.c_char * (1 << 20))()
    a = (C.addressof(buf) + 255) // 256 * 256
    assert lib.qe_gemm_fp8_ex(a, 0, 0, a, 0, 1, 256, 256, 256, a, a, a, 0, a, a, None) == 0 and lib.fake_encodes() == 3
    lib.fake_reset()
    d = qe.qe_gemm_desc(a, a, a, a, a, a, 0, 0, 0, 0, 256, 256, 256, 0)
    assert lib.qe_gemm_fp8_group((qe.qe_gemm_desc * 3)(d, d, d), 3, a, None) == 0 and lib.fake_encodes() == 9


@pytest.mark.parametrize("tokens,sums", [(256, True), (2048, True), (2688, True), (2816, False), (4096, False)])
def test_step_sums_weight_gradients_where_three_products_fit(lib, tokens, sums):
    s = fake_runtime.Stage(lib, [(256, 256)] * 2, T=tokens, M=6, slots=6)
    lib.fake_reset()
    acts = [a for a in _actions(6, 2) if a[0] != "dW"] + [("dW", l, m) for m in range(6) for l in (1, 0)]
    assert s.step(acts) == 0
    words = [w.split() for w in lib.fake_log().decode().splitlines() if " gemm " in w]  # launch STREAM gemm N products P
    assert sum(int(w[5]) for w in words) == len(acts)
    assert any(int(w[5]) > int(w[3]) for w in words) == sums
    s.close()


def test_step_takes_all_layers_of_a_unit_at_once_only_where_its_tensors_are_apart(lib):
    """Forty linears in one round, cast by one launch, their eighty GEMMs in two; as soon as one tensor that an action writes overlaps
    what another reads or writes, or a weight, or a gradient, the layers go one after the other."""
    n, M, K = 40, 2, 256
    s = fake_runtime.Stage(lib, [(K, K)] * n, M=M, slots=M, window=4)
    size = 2 * s.T * K
    base = s.buffer(4 * n * M * size)
    own = lambda l, m: [base + ((l * M + m) * 4 + j) * size for j in range(4)]  # noqa: E731
    acts = [a for a in _actions(M, n)]

    def casts(io):
        lib.fake_reset()
        assert s.step(acts, apart=io) == 0
        for h in s.layers:
            assert lib.qe_optimizer_boundary(h, M) == 0
        return max(int(w.split()[3]) for w in lib.fake_log().decode().splitlines() if " cast " in w)

    assert casts(own) == 2 * n  # the second forward and the first input gradient of every layer; the weights' casts are n
    words = [w.split() for w in lib.fake_log().decode().splitlines() if " gemm " in w]
    assert max(int(w[3]) for w in words) == n and sum(int(w[5]) for w in words) == 3 * n * M
    where = {"y on another x": (3, 1, 7, 0, 0), "dx on another dy": (3, 1, 7, 0, 2), "y on another y": (3, 1, 7, 1, 1), "dx on its own x": (3, 3, 3, 0, 0)}
    for name, (l, j, l2, m2, j2) in where.items():
        def io(a, b):
            t = own(a, b)
            if (a, b) == (l, 0):
                t[j] = own(l2, m2)[j2] + (0 if l2 == l else size - 16)
            return t
        assert casts(io) < 2 * n, name
    for name, at in (("weight", s.weights[9]), ("gradient", s.grad + 4 * s.offsets[5])):
        assert casts(lambda a, b: own(a, b)[:1] + [at - size + 16] + own(a, b)[2:] if (a, b) == (3, 0) else own(a, b)) < 2 * n, name
    s.close()


@pytest.mark.parametrize("slots", [1, 2, 3, 4, 7])
def test_step_casts_overlap_the_gemms_before_them_unless_those_read_the_slot(lib, slots):
    """The casts of a round may run beside the GEMMs of the one before, except the first round's and those of a forward into a
    slot that a weight gradient of the round before releases."""
    from paper_2609_23536_b200 import binding as qe

    M, n = 7, 3
    s = fake_runtime.Stage(lib, [(256, 256)] * n, M=M, slots=slots, window=4)
    size = 2 * s.T * 256
    base = s.buffer(4 * n * M * size)
    lib.fake_reset()
    assert s.step(_actions(M, n), apart=lambda l, m: [base + ((l * M + m) * 4 + j) * size for j in range(4)]) == 0
    casts = [w.split() for w in lib.fake_log().decode().splitlines() if " cast " in w][1:]  # (the weights' come first)
    want, free, held, last = [], set(range(slots)), {}, set()
    for r, g in enumerate(qe.plan_rounds(_actions(M, n), n, M, slots, 4, 100, max_sum=8, apart=True)):
        mine = [(a, m) for a, l, m in g if l == 0]  # the layers go alike
        for a, m in mine:
            if a == "F":
                held[m] = min(free)
                free.remove(held[m])
        if any(a != "dW" for a, m in mine):
            want.append(r > 0 and not any(a == "F" and held[m] in last for a, m in mine))
        last = {held[m] for a, m in mine if a == "dW"}
        free |= last
    assert ["early" in w for w in casts] == want and any(want) and (slots == 7 or not all(want[1:]))
    s.close()


@pytest.mark.parametrize("T,pieces", [(256, 1), (1024, 2), (2048, 4), (640, 2)])
@pytest.mark.parametrize("own_stream", [True, False], ids=["callers-stream", "execution-stream"])
def test_host_buffers_go_through_copies_and_kernels_in_pieces_of_rows(lib, T, pieces, own_stream):
    """Every row once in each direction; a piece's kernels after its upload, its read-back after its kernels, and neither waits for
    the read-back of the piece before; the caller's stream after all of them, also where a launch in the middle fails."""
    import ctypes as C

    from paper_2609_23536_b200 import binding as qe

    K, N = 256, 2048
    s = fake_runtime.Stage(lib, [(K, N)], T=T, host_io=True, slots=3, exec_stream=None if own_stream else fake_runtime.CALLER)
    x, y, tape = s.buffer(2 * T * K), s.buffer(2 * T * (N + K)), qe.qe_tape()
    assert lib.qe_forward_host(s.layers[0], 0, 0, x, y, fake_runtime.CALLER, C.byref(tape)) == 0  # (with the weight's cast)
    lib.fake_reset()
    assert lib.qe_forward_host(s.layers[0], 1, 0, x, y, fake_runtime.CALLER, C.byref(tape)) == 0
    order = fake_runtime.Order(lib.fake_log().decode())
    up, down, run = order.of("h2d"), order.of("d2h"), order.of("launch")
    assert (len(up), len(down), len(run)) == (pieces, pieces, 2 * pieces)
    for ops, at, base, row in ((up, 1, x, 2 * K), (down, 0, y, 2 * N)):  # (words of a copy: destination, source, bytes)
        parts = sorted((int(o[2][at]) - base, int(o[2][2])) for o in ops)
        assert [a for a, n in parts] == [0] + [a + n for a, n in parts][:-1] and sum(n for a, n in parts) == T * row
    for i in range(pieces):
        assert order.before(up[i], run[2 * i]) and order.before(run[2 * i + 1], down[i]) and order.seen_by(fake_runtime.CALLER, down[i])
        if i:
            assert not order.before(down[i - 1], run[2 * i]) and not order.before(down[i - 1], up[i])
    lib.fake_reset()  # an output that overlaps the input: not before all of that is up
    assert lib.qe_backward_dI_host(s.layers[0], C.byref(tape), y, y + 2 * T * N - 64, fake_runtime.CALLER) == 0
    order = fake_runtime.Order(lib.fake_log().decode())
    assert len(order.of("h2d")) == len(order.of("d2h")) == 1
    assert lib.qe_forward_host(s.layers[0], 2, 0, x, y, fake_runtime.CALLER, C.byref(tape)) == 0
    lib.fake_reset()
    lib.fake_fail(b"cudaLaunchKernelExC", 2 * pieces)
    assert lib.qe_backward_dI_host(s.layers[0], C.byref(tape), y, x, fake_runtime.CALLER) == CUDA
    order = fake_runtime.Order(lib.fake_log().decode())
    assert all(order.seen_by(fake_runtime.CALLER, o) for o in order.of("launch") + order.of("d2h"))
    s.close()


def test_no_upload_of_a_call_waits_for_its_own_read_back_however_many_calls_were_before(lib):
    import ctypes as C

    from paper_2609_23536_b200 import binding as qe

    T, K, N, pieces = 1536, 256, 2048, 3
    s = fake_runtime.Stage(lib, [(K, N)], T=T, host_io=True, slots=2, exec_stream=fake_runtime.CALLER)
    x, ys, tape = s.buffer(2 * T * K), s.buffer(4 * T * N), qe.qe_tape()
    lib.fake_reset()
    for i in range(300):  # (outputs in turn, so that they do not follow one another)
        assert lib.qe_forward_host(s.layers[0], 0, 0, x, ys + (i % 2) * 2 * T * N, fake_runtime.CALLER, C.byref(tape)) == 0
        assert lib.qe_abort_step(s.layers[0]) == 0 and lib.qe_arena_rebuild(s.layers[0]) == 0
    order = fake_runtime.Order(lib.fake_log().decode())
    up, down = order.of("h2d"), order.of("d2h")
    assert len(up) == len(down) == 300 * pieces
    assert not any(order.before(down[j], up[i]) for i in range(len(up)) for j in range(i - i % pieces, i))
    s.close()


@pytest.mark.parametrize("which", ["none", "input", "output", "unknown"])
def test_host_buffers_that_are_not_pinned_go_through_in_one_piece(lib, which):
    """A copy from or to pageable memory ends before the call that starts it does: pieces would only add waits."""
    import ctypes as C

    from paper_2609_23536_b200 import binding as qe

    T, K, N = 2048, 256, 2048
    s = fake_runtime.Stage(lib, [(K, N)], T=T, host_io=True, slots=2)
    x, y, tape = s.buffer(2 * T * K), s.buffer(2 * T * N), qe.qe_tape()
    for forward in (True, False):
        a, b, bytes_of = (x, y, {x: 2 * T * K, y: 2 * T * N}) if forward else (y, x, {x: 2 * T * K, y: 2 * T * N})
        lib.fake_reset()
        if which in ("input", "output"):
            p = a if which == "input" else b
            lib.fake_pageable(p, p + bytes_of[p])
        if which == "unknown":
            lib.fake_fail(b"cudaPointerGetAttributes", 1)
        if forward:
            assert lib.qe_forward_host(s.layers[0], 0, 0, a, b, fake_runtime.CALLER, C.byref(tape)) == 0
        else:
            assert lib.qe_backward_dI_host(s.layers[0], C.byref(tape), a, b, fake_runtime.CALLER) == 0
        order = fake_runtime.Order(lib.fake_log().decode())
        assert len(order.of("h2d")) == len(order.of("d2h")) == (4 if which == "none" else 1)
    s.close()


@pytest.mark.parametrize("mode", [0, 1], ids=["eager", "graph"])
def test_casts_that_overlap_go_ahead_on_a_count_of_commits(lib, mode):
    """A cast that does not wait for the GEMM launch before it is told how many problems will have committed by then, and that
    launch counts its own: numbers that go on from call to call, or start anew in every graph, whose last launch sets the count
    back.  Nothing counts for a cast that waits."""
    M, n = 12, 20
    s = fake_runtime.Stage(lib, [(256, 256)] * n, M=M, slots=6, mode=mode, window=4)
    size = 2 * s.T * 256
    base = s.buffer(4 * n * M * size)
    total = early = 0
    for _ in range(3):
        lib.fake_reset()
        assert s.step(_actions(M, n), apart=lambda l, m: [base + ((l * M + m) * 4 + j) * size for j in range(4)]) == 0
        for h in s.layers:
            assert lib.qe_optimizer_boundary(h, M) == 0
        log = (lib.fake_replayed() if mode else lib.fake_log()).decode()
        for piece in log.split("graph\n")[1:] if mode else [log]:
            launches = [w.split() for w in piece.splitlines() if " cast " in w or " gemm " in w]
            start = total
            for before, w in zip([[]] + launches, launches):
                if "early" in w:
                    assert before[2] == "gemm" and before[-1] == "announces"
                    total += int(before[3])
                    assert int(w[-1]) == total
                    early += 1
                else:
                    assert "announces" not in before
            assert [("withdraws" in w) for w in launches] == [False] * (len(launches) - 1) + [mode == 1 and total > start]
            total = total if mode == 0 else 0
    assert early > 15
    lib.fake_reset()
    lib.fake_fail(b"cudaGraphLaunch" if mode else b"cudaLaunchKernelExC", 2 if mode else 30)  # some of the counting is lost
    own = lambda l, m: [base + ((l * M + m) * 4 + j) * size for j in range(4)]  # noqa: E731
    assert s.step(_actions(M, n), apart=own) == CUDA and all(lib.qe_arena_rebuild(h) == 0 for h in s.layers)
    lib.fake_reset()
    assert s.step(_actions(M, n), apart=own) == 0 and b"early" not in lib.fake_log() + lib.fake_replayed()
    s.close()


@pytest.mark.parametrize("pairs,launches", [(74, 1), (73, 4), (10, 4), (0, 4)])
def test_chains_go_out_one_by_one_where_the_device_does_not_hold_all_their_blocks(lib, pairs, launches):
    import ctypes as C

    from paper_2609_23536_b200 import binding as qe

    lib.fake_pairs(pairs)
    s = fake_runtime.Stage(lib, [(256, 256)] * 4)
    lib.fake_pairs(74)
    x, y, tapes = s.buffer(2 * s.T * 256), s.buffer(2 * s.T * 256), (qe.qe_tape * 4)()
    hs = (C.c_void_p * 4)(*[h.value for h in s.layers])
    for call in (lambda: lib.qe_forward_chain(hs, 4, 0, 0, x, y, fake_runtime.CALLER, tapes),
                 lambda: lib.qe_backward_dI_chain(hs, tapes, 4, y, x, fake_runtime.CALLER)):
        lib.fake_reset()
        assert call() == 0
        words = [w.split() for w in lib.fake_log().decode().splitlines() if " gemm " in w]  # launch STREAM gemm N products P
        assert [int(w[3]) for w in words] == ([4] if launches == 1 else [1] * launches)
    s.close()


@pytest.mark.parametrize("sms", [20, 57, 148])
def test_launches_that_commit_scales_hold_a_problem_per_cta_at_most(lib, tmp_path, sms):
    """A problem's early commit is made by the CTA of its number: a device of few SMs gets more launches, not lost commits."""
    import shutil

    lib = fake_runtime.load(shutil.copy(lib._name, tmp_path / "few_sms.so"))
    lib.fake_sms(sms)
    n, M = 57, 2
    s = fake_runtime.Stage(lib, [(256, 256)] * n, M=M, slots=M, window=4)
    size = 2 * s.T * 256
    base = s.buffer(4 * n * M * size)
    lib.fake_reset()
    assert s.step(_actions(M, n), apart=lambda l, m: [base + ((l * M + m) * 4 + j) * size for j in range(4)]) == 0
    words = [w.split() for w in lib.fake_log().decode().splitlines() if " gemm " in w]  # launch STREAM gemm N products P
    assert max(int(w[3]) for w in words) <= min(56, sms // 2 * 2) and sum(int(w[5]) for w in words) == 3 * n * M
    s.close()


@pytest.mark.parametrize("n,M,w,d", [(56, 2, 2, 0), (57, 2, 2, 0), (100, 4, 1, 1), (112, 2, 1, 0), (113, 2, 1, 0)])
def test_launches_of_a_round_hold_fifty_six_problems_and_split_evenly(lib, n, M, w, d):
    """A round has 112 forwards and input gradients at most; what does not fit one launch goes out in launches of about the same
    size, weight gradients then in launches of their own."""
    from paper_2609_23536_b200 import binding as qe
    from paper_2609_23536_b200.schedules import peak_live, sched

    s = sched(M, w, d)
    acts = [(a, l, m) for a, m in s for l in (range(n) if a == "F" else range(n - 1, -1, -1))]
    stage = fake_runtime.Stage(lib, [(256, 256)] * n, T=256, M=M, slots=peak_live(s), window=4)
    size = 2 * 256 * 256
    base = stage.buffer(4 * n * M * size)
    lib.fake_reset()
    assert stage.step(acts, apart=lambda l, m: [base + ((l * M + m) * 4 + j) * size for j in range(4)]) == 0
    got = [tuple(map(int, w.split()[3:6:2])) for w in lib.fake_log().decode().splitlines() if " gemm " in w]
    stage.close()
    rounds, want = qe.plan_rounds(acts, n, M, peak_live(s), 4, 112, max_sum=8, apart=True), []

    def shares(k):
        launches = -(-k // 56)
        return [k // launches + (i < k % launches) for i in range(launches)]

    for g in rounds:
        chain = sum(a != "dW" for a, l, m in g)
        sums = {l: sum((a, x) == ("dW", l) for a, x, m in g) for a, l, m in g if a == "dW"}
        if chain + len(sums) <= 56:
            want.append((chain + len(sums), len(g)))
        else:
            want += [(k, k) for k in shares(chain)]
            products = set(sums.values())
            assert len(products) < 2
            want += [(k, k * max(products)) for k in shares(len(sums))] if sums else []
    assert got == want
    assert {56: want[0] == (56, 56), 57: want[:2] == [(29, 29), (28, 28)], 100: (50, 50) in want, 112: want[-2:] == [(56, 112)] * 2,
            113: (1, 1) not in want and max(want) < (57, 0)}[n]
