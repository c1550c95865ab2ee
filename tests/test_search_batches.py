"""awq_search_alpha evaluates several grid points per launch: the losses against those of the library's own calls, one
grid point at a time, where batches, rows and channels are ragged; and the scratch that this takes."""
import ctypes

import numpy as np
import pytest


def _one_point_bytes(M, N, K, G):
    """s, x / s, the packed arrays, y, the reference product, 1024 partial sums in fp64, 64 losses: each from a multiple of 256."""
    parts = (K * 4, M * K * 2, N * K // 2, K // G * N * 2, K // G * N // 2, M * N * 2, M * N * 4, 1024 * 8, 64 * 4)
    return sum((b + 255) // 256 * 256 for b in parts)


def test_scratch_sizes():
    from paper_2306_00978_b200 import binding, build
    build.build()
    L = binding.lib()
    for M, N, K, G in ((512, 4096, 4096, 128), (1, 128, 128, 64), (97, 384, 640, 64), (1000, 8192, 8192, 128)):
        one = L.awq_search_scratch_bytes(M, N, K, G)
        assert 0 < one <= _one_point_bytes(M, N, K, G)
        sizes = [L.awq_search_scratch_bytes_points(M, N, K, G, n) for n in range(1, 65)]
        assert sizes[0] == one and sizes == sorted(sizes)
        assert sizes[-1] <= max(one, (384 << 20) + M * N * 4)
    assert L.awq_search_scratch_bytes_points(512, 4096, 4096, 128, 20) >= 20 * 512 * 4096 * 4
    assert L.awq_search_scratch_bytes_points(16, 256, 2048, 256, 4) == 0
    assert L.awq_search_scratch_bytes_points(16, 256, 2048, 128, 0) == L.awq_search_scratch_bytes_points(16, 256, 2048, 128, 65) == 0


def _inputs(N, K, M):
    import torch
    gen = torch.Generator(device="cuda")
    gen.manual_seed(N + K + M)
    W = (torch.randn(N, K, generator=gen, device="cuda") * 0.02).half()
    X = torch.randn(M, K, generator=gen, device="cuda")
    X[:, :: max(1, K // 16)] *= 20.0
    X = X.half()
    return W, X, X.float().abs().mean(dim=0)


@pytest.mark.gpu
@pytest.mark.parametrize("N,K,M,G,n", [(512, 1024, 97, 128, 7), (384, 640, 200, 128, 3), (512, 1024, 20, 64, 4), (256, 128, 65, 64, 1)])
@pytest.mark.parametrize("points", [1, 2, 64])
def test_any_scratch_that_holds_a_grid_point(N, K, M, G, n, points):
    """Grid points are evaluated one by one, by two or all together as the scratch allows, and nothing is written behind it."""
    import torch
    from paper_2306_00978_b200 import binding
    L = binding.lib()
    W, X, stat = _inputs(N, K, M)
    alphas = [float(np.float32(i / n)) for i in range(n)]
    want, best = binding.search_alpha(W, stat, X, G, alphas)
    size = L.awq_search_scratch_bytes_points(M, N, K, G, points)
    buf = torch.full((size + 4096,), 0xA5, dtype=torch.uint8, device="cuda")
    a, losses, index = (ctypes.c_float * n)(*alphas), (ctypes.c_float * n)(), ctypes.c_int(-1)

    def call(nbytes):
        return L.awq_search_alpha(W.data_ptr(), stat.data_ptr(), X.data_ptr(), M, N, K, G, a, n, losses, ctypes.byref(index),
                                  buf.data_ptr(), nbytes, torch.cuda.current_stream().cuda_stream)

    assert call(L.awq_search_scratch_bytes(M, N, K, G) - 1) == 10
    assert call(size) == 0
    binding.poll_status()
    assert bool((buf[size:] == 0xA5).all())
    # a product by itself may add its fp32 sums in another order: 2^-10 of an fp16 output here and there
    assert np.allclose(list(losses), want, rtol=1e-3) and index.value == best


@pytest.mark.gpu
def test_a_search_near_the_memory_limit(monkeypatch):
    """Where the scratch for all grid points cannot be had, fewer are evaluated together."""
    import torch
    from paper_2306_00978_b200 import binding
    N, K, M, G, n = 512, 1024, 97, 128, 10
    W, X, stat = _inputs(N, K, M)
    alphas = [i / n for i in range(n)]
    want, best = binding.search_alpha(W, stat, X, G, alphas)
    limit, real, asked = binding.lib().awq_search_scratch_bytes_points(M, N, K, G, 2), torch.empty, []

    def empty(size, **kw):
        asked.append(size)
        if size > limit:
            raise torch.OutOfMemoryError("out of memory")
        return real(size, **kw)

    monkeypatch.setattr(torch, "empty", empty)
    losses, index = binding.search_alpha(W, stat, X, G, alphas)
    assert len(asked) == 3 and asked[-1] <= limit
    assert np.allclose(losses, want, rtol=1e-3) and index == best
    monkeypatch.setattr(torch, "empty", lambda size, **kw: (_ for _ in ()).throw(torch.OutOfMemoryError("out of memory")))
    with pytest.raises(torch.OutOfMemoryError):
        binding.search_alpha(W, stat, X, G, alphas)


@pytest.mark.gpu
@pytest.mark.parametrize("N,K,M,G,n", [
    (256, 128, 65, 64, 3),          # all points in one launch, one token past a tile
    (512, 1152, 97, 128, 64),       # the longest list, rows padded to 128
    (1536, 2048, 24, 128, 64),      # the quantizer's blocks hold so many arrays of scales that three of them fit an SM
    (2048, 2048, 24, 128, 64),      # and would, but parts of half the arrays fill the SMs better
    (384, 640, 200, 128, 5),        # an odd number of 128-channel slabs: one launch per point
    (512, 1024, 20, 64, 4),         # few tokens: the layer's own kernel per point
    (4096, 8192, 900, 128, 11),     # two batches, of six and five
])
def test_losses_are_those_of_single_calls(N, K, M, G, n):
    import torch
    from paper_2306_00978_b200 import binding
    W, X, stat = _inputs(N, K, M)
    alphas = [float(np.float32(i / n)) for i in range(n)]
    losses, best = binding.search_alpha(W, stat, X, G, alphas)
    target = X.double() @ W.double().t()
    want, slack = [], []
    for alpha in alphas:
        s = binding.channel_scale(stat, alpha, K)
        y = binding.linear((X.float() / s).half(), *binding.quantize_pack(W, stat, alpha, G), N, K, G).double()
        e = (y - target).abs()
        # another order of the fp32 sums moves an fp16 output by at most one unit in its last place (2^-10 of it), the
        # reference product in fp32 by K * 2^-24 of sum |X||W| <= 1e-3 of e here at the very most
        u = y.abs() * 2.0 ** -10 + e * 1e-3 + 2.0 ** -24
        want.append(float((e * e).mean()))
        slack.append(float((2 * e * u + u * u).mean()))
    binding.poll_status()
    got = np.asarray(losses, dtype=np.float64)
    assert (np.abs(got - want) <= np.asarray(slack)).all(), (got / np.asarray(want)).round(5)
    assert got[best] == got.min()
