"""The SM-pair prefill kernel (asked for by name: up to 256 tokens awq_linear may take the stream kernel): its tile widths (64, 128,
192, 256 tokens), an odd last slab of 128 channels and tiles cut by stream-K, against the fp64 oracle."""
import numpy as np
import pytest

from tests.test_workspace_rules import _NoWorkspace
from tests.util import Case, assert_parity, oracle_packed_to_cuda, to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M,G,cut", [
    (256, 128, 65, 128, False),          # one stage, one token past a 64-token tile
    (384, 256, 130, 64, False),          # an absent second slab in the last pair
    (128, 640, 129, 128, False),         # nothing but half a pair
    (4096, 256, 333, 128, False),        # 128-token tiles: with 64 there would be two waves
    (4224, 1024, 700, 64, False),        # 192-token tiles, odd number of slabs
    (4096, 2048, 1000, 128, False),      # 256-token tiles
    (2816, 8192, 130, 128, True),        # 64-token tiles, K loops cut over the pairs
    (1152, 8192, 300, 64, True),         # the same with an odd slab, groups of 64, tiles in up to four parts
    (512, 8192, 520, 128, True),
])
def test_tile_widths(N, K, M, G, cut):
    from paper_2306_00978_b200 import binding
    case = Case(5300 + N + K + M, N, K, M, G, 0.5)
    packed = oracle_packed_to_cuda(case)
    x = to_cuda(case.x)
    y = binding.linear(x, *packed, N, K, G, path=binding.PATH_GEMM)
    n0 = binding.launch_count()
    again = binding.linear(x, *packed, N, K, G, path=binding.PATH_GEMM)
    assert binding.launch_count() - n0 == 1
    binding.poll_status()
    assert_parity(y.cpu().numpy(), case.y_ref(), f"N={N} K={K} M={M} G={G}")
    assert np.array_equal(y.cpu().numpy().view(np.uint16), again.cpu().numpy().view(np.uint16))
    with _NoWorkspace():                 # whole tiles: the sums of a cut tile are formed in another order
        whole = binding.lib().awq_linear_path(x.data_ptr(), *(t.data_ptr() for t in packed), again.data_ptr(), M, N, K, G,
                                              binding.PATH_GEMM, None)
        assert whole == 0
    assert bool((y == again).all()) == (not cut)


@pytest.mark.parametrize("N,K,M,one_sm", [
    (256, 13824, 100, True),      # a tile's K loop over 16 SMs
    (640, 13824, 65, True),
    (256, 8192, 128, True),
    (256, 1024, 100, False),      # short rows
    (1280, 13824, 100, False),    # too many tiles for 16 SMs each
])
def test_few_channels_and_65_to_128_tokens(N, K, M, one_sm):
    """Among the prefill kernels, few channels and long rows at 65 .. 128 tokens run on the one-SM kernel, whose sums are formed in
    another order than the SM-pair kernel's; awq_linear leaves it these shapes."""
    from paper_2306_00978_b200 import binding
    case = Case(5900 + N + K + M, N, K, M, 128, 0.5)
    packed = oracle_packed_to_cuda(case)
    x = to_cuda(case.x)
    auto = binding.linear(x, *packed, N, K, 128)
    y = binding.linear(x, *packed, N, K, 128, path=binding.PATH_GEMM)
    forced = binding.linear(x, *packed, N, K, 128, path=binding.PATH_GEMM_1SM)
    binding.poll_status()
    assert_parity(y.cpu().numpy(), case.y_ref(), f"N={N} K={K} M={M}")
    assert_parity(auto.cpu().numpy(), case.y_ref(), f"automatic, N={N} K={K} M={M}")
    assert bool((y == forced).all()) == one_sm
    if one_sm:
        assert bool((auto == forced).all())
