"""The clip search rules ratios out by estimates and evaluates as defined only what is left: groups where that is decided by the
last bits (equal ratios, all-zero and constant groups, weights on the grid) or cannot be (a range far from zero, infinities,
not-a-number), odd numbers of ratios, and enough random groups to meet near ties.  The chosen ratios are the oracle's."""
import numpy as np
import pytest

from oracle import awq_oracle as orc
from tests.util import to_cuda

pytestmark = pytest.mark.gpu


def _groups(N, K, G, seed):
    rng = np.random.default_rng(seed)
    W = (rng.standard_normal((N, K)) * 0.02).astype(np.float16)
    g = W.reshape(N, K // G, G)
    kind = rng.integers(0, 24, (N, K // G))
    g[kind == 0] = 0.0
    g[kind == 1] = 0.375
    g[kind == 2] = (rng.integers(0, 16, (int((kind == 2).sum()), G)) / 64.0).astype(np.float16)
    g[kind == 3] = (rng.integers(0, 8, (int((kind == 3).sum()), G)) / 64.0 - 0.0625).astype(np.float16)
    g[kind == 4] = (1000.0 + rng.integers(0, 2, (int((kind == 4).sum()), G)) * 0.5).astype(np.float16)
    g[kind == 5] = (rng.standard_normal((int((kind == 5).sum()), G)) * 6e-8).astype(np.float16)      # subnormal
    g[kind == 6] = (rng.standard_normal((int((kind == 6).sum()), G)) * 1e4).astype(np.float16)
    g[kind == 7, 3] = np.float16(np.inf)
    g[kind == 8, 5] = np.float16(-np.inf)
    g[kind == 9, 7] = np.float16(np.nan)
    g[kind == 10] = np.abs(g[kind == 10])
    return W


@pytest.mark.parametrize("N,K,G,bits", [(256, 1024, 128, 4), (256, 1024, 64, 3), (1024, 4096, 128, 3)])
@pytest.mark.parametrize("ratios", [[1.0], [1.0, 0.9, 0.9, 1.0, 0.8, 0.8, 0.8], [1.0 - 0.5 * i / 32 for i in range(32)],
                                    [1.0 - 1e-6 * i for i in range(9)], [0.5 + 0.05 * i for i in range(11)],
                                    [0.9, 1.0], [0.7, 0.85, 0.85], [1.0, 1.0 - 1e-6, 0.8, 0.8], [0.6, 0.7, 0.8, 0.9, 1.0]], ids=len)
@pytest.mark.parametrize("scaled", [False, True])
def test_ratios_are_the_defined_ones(N, K, G, bits, ratios, scaled):
    from paper_2306_00978_b200 import binding
    ratios = [float(np.float32(r)) for r in ratios]
    W = _groups(N, K, G, N + K + G + len(ratios))
    stat = (np.abs(np.random.default_rng(bits).standard_normal(K)) + 0.05).astype(np.float32)
    alpha = 0.5 if scaled else 0.0
    with np.errstate(all="ignore"):
        want = orc.search_clip(W, orc.channel_scale(stat, alpha), G, ratios, bits=bits)
    got = binding.search_clip(to_cuda(W), to_cuda(stat), alpha, G, ratios, bits=bits).cpu().numpy()
    bad = np.argwhere(got.view(np.uint32) != want.view(np.uint32))
    assert len(bad) == 0, (len(bad), bad[:5].tolist())
