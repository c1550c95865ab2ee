"""The quantizer where a thread block's range of tiles crosses column blocks, and on weights that sit on ties of the
rounding, which take its element-by-element path: packed words, zero points and scales bit-identical to the oracle's."""
import numpy as np
import pytest

from oracle import awq_oracle as orc
from tests.util import to_cuda

pytestmark = pytest.mark.gpu


def _weights(N, K, G, ties, seed):
    rng = np.random.default_rng(seed)
    W = (rng.standard_normal((N, K)) * 0.02).astype(np.float16)
    if ties:
        # levels of half a step: min 0 or -7, max 15 or 8 steps of 2^-6, so every odd level is a quotient k + 1/2
        tied = rng.integers(0, 31, (N, K // G, G)) / 2.0
        tied[:, :, 0], tied[:, :, 1] = 0.0, 15.0
        tied -= rng.choice([0.0, 7.0], (N, K // G, 1))
        half = rng.random((N, K // G)) < 0.5
        W.reshape(N, K // G, G)[half] = (tied[half] * 2.0 ** -6).astype(np.float16)
    return W


# more tiles than resident blocks (4 per SM of 128 threads, 2 of 256), in numbers that do not divide
@pytest.mark.parametrize("N,K,G", [(1152, 5376, 64), (1152, 5376, 128), (1152, 5376, 256), (1408, 5632, 512), (2048, 5120, 1024), (128, 128, 128)])
@pytest.mark.parametrize("bits,symmetric,clipped", [(4, False, False), (3, True, False), (4, False, True)])
def test_ranges_and_ties(N, K, G, bits, symmetric, clipped):
    from paper_2306_00978_b200 import binding
    W = _weights(N, K, G, True, N + K + G + bits)
    stat = (np.abs(np.random.default_rng(G).standard_normal(K)) + 0.25).astype(np.float32)
    clip = np.random.default_rng(K).choice(np.float32([1.0, 0.75, 0.55]), (N, K // G)).astype(np.float32) if clipped else None
    for alpha in (0.0, float(np.float32(0.35))):                # (alpha is an fp32 argument)
        qw, sc, zp = binding.quantize_pack(to_cuda(W), to_cuda(stat), alpha, G, bits=bits, symmetric=symmetric,
                                           clip_ratio=None if clip is None else to_cuda(clip))
        want = orc.quantize_pack(W, stat, alpha, G, clip=clip, bits=bits, symmetric=symmetric)
        assert np.array_equal(qw.cpu().numpy().view(np.uint32).reshape(-1), want[0])
        assert np.array_equal(sc.cpu().numpy().view(np.uint16).reshape(-1), want[1].view(np.uint16).reshape(-1))
        assert np.array_equal(zp.cpu().numpy().view(np.uint8).reshape(-1), want[2].reshape(-1))
