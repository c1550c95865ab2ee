"""awq_search_alpha evaluates several grid points per launch: the losses against those of the library's own calls, one
grid point at a time, where batches, rows and channels are ragged."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M,G,n", [
    (256, 128, 65, 64, 3),          # all points in one launch, one token past a tile
    (512, 1152, 97, 128, 64),       # the longest list, rows padded to 128
    (384, 640, 200, 128, 5),        # an odd number of 128-channel slabs: one launch per point
    (512, 1024, 20, 64, 4),         # few tokens: the layer's own kernel per point
    (4096, 8192, 900, 128, 11),     # two batches, of six and five
])
def test_losses_are_those_of_single_calls(N, K, M, G, n):
    import torch
    from paper_2306_00978_b200 import binding
    gen = torch.Generator(device="cuda")
    gen.manual_seed(N + K + M)
    W = (torch.randn(N, K, generator=gen, device="cuda") * 0.02).half()
    X = torch.randn(M, K, generator=gen, device="cuda")
    X[:, :: max(1, K // 16)] *= 20.0
    X = X.half()
    stat = X.float().abs().mean(dim=0)
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
