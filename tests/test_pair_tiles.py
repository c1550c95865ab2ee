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


@pytest.mark.parametrize("N,K,M,one_sm", [
    (256, 13824, 100, True),      # a tile's K loop over 16 SMs
    (640, 13824, 65, True),
    (256, 8192, 128, True),
    (256, 1024, 100, False),      # short rows
    (1280, 13824, 100, False),    # too many tiles for 16 SMs each
])
def test_few_channels_and_65_to_128_tokens(N, K, M, one_sm):
    """Few channels and long rows at 65 .. 128 tokens run on the one-SM kernel, whose sums are formed in another
    order than the SM-pair kernel's."""
    from paper_2306_00978_b200 import binding
    case = Case(5900 + N + K + M, N, K, M, 128, 0.5)
    packed = oracle_packed_to_cuda(case)
    x = to_cuda(case.x)
    y = binding.linear(x, *packed, N, K, 128)
    forced = binding.linear(x, *packed, N, K, 128, path=binding.PATH_GEMM_1SM)
    binding.poll_status()
    assert_parity(y.cpu().numpy(), case.y_ref(), f"N={N} K={K} M={M}")
    assert bool((y == forced).all()) == one_sm
