"""Calls on several streams and threads: a layer call behind a writer of its packed arrays waits for it whatever runs elsewhere
on the device, and calls that need no workspace may overlap.  How a launch is ordered behind the one in front is read from the
edges of a captured graph, which is not launched."""
import contextlib
import ctypes
import threading

import numpy as np
import pytest

from tests.util import Case, oracle_packed_to_cuda, to_cuda

pytestmark = pytest.mark.gpu

FULL, PROGRAMMATIC = 0, 1                # cudaGraphDependencyType


class _EdgeData(ctypes.Structure):
    _fields_ = [("from_port", ctypes.c_ubyte), ("to_port", ctypes.c_ubyte), ("type", ctypes.c_ubyte), ("reserved", ctypes.c_ubyte * 5)]


@contextlib.contextmanager
def _captured_edges(stream):
    """Captures what is enqueued on `stream` inside; yields a list that holds the edges' types afterwards, in stream order."""
    rt = ctypes.CDLL("libcudart.so.12")
    ptr, size, types = ctypes.c_void_p, ctypes.c_size_t, []
    handle, graph, n = ptr(stream.cuda_stream), ptr(), size()
    assert rt.cudaStreamBeginCapture(handle, 2) == 0                      # relaxed: other streams go on as before
    try:
        yield types
    finally:
        assert rt.cudaStreamEndCapture(handle, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetEdges_v2(graph, None, None, None, ctypes.byref(n)) == 0
    begin, end, data = (ptr * n.value)(), (ptr * n.value)(), (_EdgeData * n.value)()
    assert rt.cudaGraphGetEdges_v2(graph, begin, end, data, ctypes.byref(n)) == 0
    follow = {b: (e, d.type) for b, e, d in zip(begin, end, data)}
    assert len(follow) == n.value                                         # a chain
    node = next(b for b in follow if b not in set(end))
    while node in follow:
        node, kind = follow[node]
        types.append(kind)
    assert rt.cudaGraphDestroy(graph) == 0


@contextlib.contextmanager
def _capture(rt, stream):
    """Captures what is enqueued on `stream` and the streams joined to it; yields a list that holds the graph's edges (from, to, type)
    afterwards."""
    ptr, size, edges = ctypes.c_void_p, ctypes.c_size_t, []
    graph, n = ptr(), size()
    assert rt.cudaStreamBeginCapture(stream, 2) == 0
    try:
        yield edges
    finally:
        assert rt.cudaStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetEdges_v2(graph, None, None, None, ctypes.byref(n)) == 0
    begin, end, data = (ptr * n.value)(), (ptr * n.value)(), (_EdgeData * n.value)()
    assert rt.cudaGraphGetEdges_v2(graph, begin, end, data, ctypes.byref(n)) == 0
    edges += [(b, e, d.type) for b, e, d in zip(begin, end, data)]
    assert rt.cudaGraphDestroy(graph) == 0


def _operands(N, K, M, G, bits=4):
    import torch
    torch.manual_seed(N + K + M)
    qw = torch.randint(0, 256, (N * K * bits // 8,), dtype=torch.uint8, device="cuda")
    sc = (torch.rand((N // 16, K // G, 16), device="cuda") * 0.01 + 0.001).half()
    zp = torch.randint(0, 256, (N // 32, K // G, 16), dtype=torch.uint8, device="cuda")
    return torch.randn((M, K), device="cuda").half(), qw, sc, zp, torch.empty((M, N), dtype=torch.float16, device="cuda")


@pytest.mark.parametrize("M,N,K", [
    (1, 8192, 4096), (5, 8192, 8320), (5, 4096, 8320),                   # band, chunked and stream kernel
    (16, 8192, 4096), (100, 8192, 4096), (300, 8192, 4096),              # stream and SM-pair kernel
])
def test_a_call_on_another_stream_does_not_release_the_reader(M, N, K):
    import torch
    from paper_2306_00978_b200 import binding
    G = 128
    L = binding.lib()
    x, qw, sc, zp, y = _operands(N, K, M, G)
    other = _operands(N, K, M, G)
    W = (torch.randn((N, K), device="cuda") * 0.02).half()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()

    def layer(stream, x, qw, sc, zp, y):
        assert L.awq_linear(x.data_ptr(), qw.data_ptr(), sc.data_ptr(), zp.data_ptr(), y.data_ptr(), M, N, K, G, stream.cuda_stream) == 0

    binding.linear(x, qw, sc, zp, N, K, G, out=y)
    torch.cuda.synchronize()
    layer(a, x, qw, sc, zp, y)
    torch.cuda.synchronize()
    with _captured_edges(a) as types:
        assert L.awq_quantize_pack(W.data_ptr(), None, 0.0, G, qw.data_ptr(), sc.data_ptr(), zp.data_ptr(), N, K, a.cuda_stream) == 0
        layer(b, *other)
        layer(a, x, qw, sc, zp, y)
        layer(a, x, qw, sc, zp, y)
    binding.poll_status()
    assert types[0] == FULL
    assert PROGRAMMATIC in types[1:]                      # only the first call behind the writer is held back


@pytest.mark.parametrize("M,others", [(1, 0), (5, 0), (16, 0), (300, 0), (1, 70)])
def test_a_captured_call_joined_behind_a_writer_on_another_stream(M, others):
    """The quantizer on a second stream of the capture; a call there that waits for it, and one joined behind the quantizer itself by an
    event, with `others` captures of a writer and its reader begun and ended in between (more than are remembered)."""
    import torch
    from paper_2306_00978_b200 import binding
    rt = ctypes.CDLL("libcudart.so.12")
    ptr = ctypes.c_void_p
    N, K, G = (8192, 4096, 128) if M != 5 else (8192, 8320, 128)
    L = binding.lib()
    x, qw, sc, zp, y = _operands(N, K, M, G)
    W = torch.zeros((N, K), dtype=torch.float16, device="cuda")
    binding.linear(x, qw, sc, zp, N, K, G, out=y)
    torch.cuda.synchronize()
    events, streams = [ptr() for _ in range(3)], [ptr() for _ in range(2 + others)]
    for e in events:
        assert rt.cudaEventCreateWithFlags(ctypes.byref(e), 2) == 0       # without timing
    for s in streams:
        assert rt.cudaStreamCreateWithFlags(ctypes.byref(s), 1) == 0      # non-blocking
    a, b = streams[:2]

    def quantize(stream):
        assert L.awq_quantize_pack(W.data_ptr(), None, 0.0, G, qw.data_ptr(), sc.data_ptr(), zp.data_ptr(), N, K, stream) == 0

    def layer(stream):
        assert L.awq_linear(x.data_ptr(), qw.data_ptr(), sc.data_ptr(), zp.data_ptr(), y.data_ptr(), M, N, K, G, stream) == 0

    def record(event, stream, waits):
        assert rt.cudaEventRecord(event, stream) == 0 and rt.cudaStreamWaitEvent(waits, event, 0) == 0

    with _capture(rt, a) as edges:
        record(events[0], a, b)
        quantize(b)
        assert rt.cudaEventRecord(events[1], b) == 0
        layer(b)
        for s in streams[2:]:
            with _capture(rt, s):
                quantize(s)
                layer(s)
        assert rt.cudaStreamWaitEvent(a, events[1], 0) == 0
        layer(a)
        layer(a)
        record(events[2], b, a)
    for s in streams:
        assert rt.cudaStreamDestroy(s) == 0
    for e in events:
        assert rt.cudaEventDestroy(e) == 0
    binding.poll_status()
    roots = {f for f, _, _ in edges} - {t for _, t, _ in edges}
    assert len(roots) == 1                                # the quantizer
    assert [kind for f, _, kind in edges if f in roots] == [FULL, FULL]


def test_the_folded_scale_behind_its_writer():
    import torch
    from paper_2306_00978_b200 import binding
    N, K, M, G = 8192, 4096, 1, 128
    L = binding.lib()
    x, qw, sc, zp, y = _operands(N, K, M, G)
    stat, inv_s = torch.rand(K, device="cuda") + 0.5, torch.empty(K, device="cuda")
    a = torch.cuda.Stream()

    def layer():
        assert L.awq_linear_scaled(x.data_ptr(), inv_s.data_ptr(), None, qw.data_ptr(), sc.data_ptr(), zp.data_ptr(), y.data_ptr(),
                                   M, N, K, G, a.cuda_stream) == 0

    torch.cuda.synchronize()
    layer()
    torch.cuda.synchronize()
    with _captured_edges(a) as types:
        assert L.awq_inverse_channel_scale(stat.data_ptr(), 0.5, inv_s.data_ptr(), K, a.cuda_stream) == 0      # two launches
        layer()
        layer()
    binding.poll_status()
    assert types == [FULL, FULL, PROGRAMMATIC]


@pytest.mark.parametrize("M", [16, 300])
def test_int3_calls_beside_another_thread(M):
    """At 16 tokens the stream kernel reads the 3-bit storage, plainly ordered, and the kernel that adds its parts may be set up meanwhile; at
    300 the storage is expanded, and expansion and reader are plainly ordered."""
    import torch
    from paper_2306_00978_b200 import binding
    N, K, G, calls = 2048, 2048, 128, 300
    L = binding.lib()
    x, qw3, sc, zp, y = _operands(N, K, M, G, bits=3)
    ox, oqw, osc, ozp, oy = _operands(N, K, M, G)
    scratch = torch.empty(N * K // 2, dtype=torch.uint8, device="cuda")
    a, b, stop = torch.cuda.Stream(), torch.cuda.Stream(), threading.Event()
    binding.linear(ox, oqw, osc, ozp, N, K, G, out=oy)
    torch.cuda.synchronize()

    def others():
        while not stop.is_set():
            for _ in range(32):
                assert L.awq_linear(ox.data_ptr(), oqw.data_ptr(), osc.data_ptr(), ozp.data_ptr(), oy.data_ptr(), M, N, K, G, b.cuda_stream) == 0
            b.synchronize()

    thread = threading.Thread(target=others)
    thread.start()
    try:
        with _captured_edges(a) as types:
            for _ in range(calls):
                assert L.awq_linear_int3(x.data_ptr(), qw3.data_ptr(), sc.data_ptr(), zp.data_ptr(), y.data_ptr(), scratch.data_ptr(),
                                         M, N, K, G, a.cuda_stream) == 0
    finally:
        stop.set()
        thread.join()
    binding.poll_status()
    per_call = (len(types) + 1) // calls                  # the expansion if there is one, the layer's kernel, and the one that adds parts if there is one
    assert per_call * calls == len(types) + 1 and per_call >= 2
    assert types[per_call - 1::per_call] == [FULL] * (calls - 1)          # from call to call
    assert types[::per_call] == [PROGRAMMATIC if M == 16 else FULL] * calls


@pytest.mark.parametrize("widths,K,M,G", [((4096, 2304), 5248, 4, 128), ((2176, 4352), 8192, 8, 64)])
def test_several_matrices_up_to_8_tokens_need_no_workspace(widths, K, M, G):
    """Long rows, many output rows: one launch of the band kernel, bit for bit what it gives each matrix alone, and nothing that two
    streams or threads would share."""
    import torch
    from paper_2306_00978_b200 import binding
    cases = [Case(6900 + i, n, K, M, G, 0.5) for i, n in enumerate(widths)]
    mats = [(*oracle_packed_to_cuda(c), c.N) for c in cases]
    inv_s = to_cuda((np.float32(1.0) / cases[0].s).astype(np.float32))
    xs = [torch.randn((M, K), device="cuda").half() for _ in range(2)]
    scaled_x = [(x.float() * inv_s).half() for x in xs]
    want = [[binding.linear(x, *m[:3], m[3], K, G, path=binding.PATH_GEMV) for m in mats] for x in xs]
    want_scaled = [[binding.linear(x, *m[:3], m[3], K, G, path=binding.PATH_GEMV) for m in mats] for x in scaled_x]
    n0 = binding.launch_count()
    plain = binding.linear_multi(xs[0], mats, K, G)
    assert binding.launch_count() - n0 == 1
    assert all(torch.equal(y, w) for y, w in zip(plain, want[0]))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in xs]
    got = [[], []]

    def calls(i):
        with torch.cuda.stream(streams[i]):
            for _ in range(40):
                got[i].append((binding.linear_multi(xs[i], mats, K, G), binding.linear_multi_scaled(xs[i], inv_s, mats, K, G)))

    threads = [threading.Thread(target=calls, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    binding.poll_status()
    for i in range(2):
        assert len(got[i]) == 40
        for plain, scaled in got[i]:
            assert all(torch.equal(y, w) for y, w in zip(plain, want[i]))
            assert all(torch.equal(y, w) for y, w in zip(scaled, want_scaled[i]))


def test_calls_from_a_thread_that_has_not_used_the_gpu():
    """Tensor maps are encoded by the driver in the thread's context, which nothing but the call itself has made current."""
    import torch
    from paper_2306_00978_b200 import binding
    N, K, G = 1024, 1024, 128
    L, n = binding.lib(), 3
    operands = [(M, *_operands(N, K, M, G)) for M in (1, 16, 100, 300)]
    for M, x, qw, sc, zp, y in operands:
        binding.linear(x, qw, sc, zp, N, K, G, out=y)
    W, X = (torch.randn((N, K), device="cuda") * 0.02).half(), torch.randn((96, K), device="cuda").half()
    stat = X.float().abs().mean(dim=0)
    alphas = [0.0, 0.5, 1.0]
    want, best = binding.search_alpha(W, stat, X, G, alphas)
    need = L.awq_search_scratch_bytes(96, N, K, G)
    scratch = torch.empty(need, dtype=torch.uint8, device="cuda")
    outs = [torch.empty_like(o[-1]) for o in operands]
    a, losses, index = (ctypes.c_float * n)(*alphas), (ctypes.c_float * n)(), ctypes.c_int(-1)
    torch.cuda.synchronize()
    calls = [lambda o=o, y=y: L.awq_linear(*(t.data_ptr() for t in o[1:5]), y.data_ptr(), o[0], N, K, G, None) for o, y in zip(operands, outs)]
    calls.append(lambda: L.awq_search_alpha(W.data_ptr(), stat.data_ptr(), X.data_ptr(), 96, N, K, G, a, n, losses, ctypes.byref(index),
                                            scratch.data_ptr(), need, None))
    status = []
    for call in calls:
        thread = threading.Thread(target=lambda: status.append(call()))
        thread.start()
        thread.join()
    binding.poll_status()
    assert status == [0] * len(calls)
    assert all(torch.equal(y, o[-1]) for y, o in zip(outs, operands))
    assert list(losses) == want and index.value == best
