"""The SM-pair prefill kernel's tile widths (64, 128, 192, 256 tokens), an odd last slab of 128 channels and
tiles cut by stream-K, against the fp64 oracle."""
import numpy as np
import pytest

from tests.util import Case, assert_parity, oracle_packed_to_cuda, to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M,G", [
    (256, 128, 65, 128),          # one stage, one token past a 64-token tile
    (384, 256, 130, 64),          # an absent second slab in the last pair
    (128, 640, 129, 128),         # nothing but half a pair
    (4096, 256, 333, 128),        # 128-token tiles: with 64 there would be two waves
    (4224, 1024, 700, 64),        # 192-token tiles, odd number of slabs
    (4096, 2048, 1000, 128),      # 256-token tiles
    (2816, 8192, 130, 128),       # 64-token tiles, K loops cut over the pairs
])
def test_tile_widths(N, K, M, G):
    from paper_2306_00978_b200 import binding
    case = Case(5300 + N + K + M, N, K, M, G, 0.5)
    packed = oracle_packed_to_cuda(case)
    y = binding.linear(to_cuda(case.x), *packed, N, K, G)
    again = binding.linear(to_cuda(case.x), *packed, N, K, G)
    binding.poll_status()
    assert_parity(y.cpu().numpy(), case.y_ref(), f"N={N} K={K} M={M} G={G}")
    assert np.array_equal(y.cpu().numpy().view(np.uint16), again.cpu().numpy().view(np.uint16))
