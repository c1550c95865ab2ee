"""The stream kernel (tiles of 256 channels x up to 128 tokens on SM pairs, their K loops laid end to end and cut into
one range per pair) where it can go wrong: widths of a token tile, tiles cut into two and into many parts, a last stage of
128 channels, an odd 128-channel slab, two token tiles, several matrices and the folded scale, against the fp64 oracle."""
import numpy as np
import pytest

from oracle import awq_oracle as orc
from paper_2306_00978_b200 import synth
from tests.test_stream_kernel_to_64_tokens import unrounded_bound
from tests.util import Case, assert_parity, oracle_packed_to_cuda, to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M,G", [
    (256, 256, 32, 128),           # one stage, one pair, nothing cut
    (19200, 256, 9, 128),          # 75 tiles of one stage for 74 pairs: still nothing to add
    (4096, 4096, 16, 128),         # each tile in four to six parts
    (2432, 1152, 17, 64),          # odd slab, last stage of 128 channels, four groups a stage
    (128, 8192, 31, 128),          # one half tile over 32 pairs
    (12288, 640, 24, 128),         # ranges of two and three stages that start inside a tile
    (512, 2176, 33, 64), (896, 4096, 47, 128), (1024, 1536, 64, 512),      # 48 and 64 tokens a tile
    (1024, 4096, 65, 128), (640, 5120, 97, 64), (2048, 8192, 128, 128),    # 80, 112, 128
    (1152, 8192, 130, 128), (384, 4224, 250, 128),                         # two token tiles
])
def test_linear(N, K, M, G):
    from paper_2306_00978_b200 import binding
    case = Case(6200 + N + K + M + G, N, K, M, G, 0.5)
    packed = oracle_packed_to_cuda(case)
    y = binding.linear(to_cuda(case.x), *packed, N, K, G)
    n0 = binding.launch_count()
    again = binding.linear(to_cuda(case.x), *packed, N, K, G)
    launches = binding.launch_count() - n0
    binding.poll_status()
    # the second launch adds the parts of cut tiles (and tells this kernel from the prefill kernels)
    assert launches == (1 if K <= 256 else 2)
    y = y.cpu().numpy()
    assert np.array_equal(y.view(np.uint16), again.cpu().numpy().view(np.uint16))
    if M <= 32:
        ref, bound = unrounded_bound(case.x, orc.dequantize(case.codes, case.zeros, case.scales, G))
        assert (np.abs(y.astype(np.float64) - ref) <= bound).all()
    else:
        assert_parity(y, case.y_ref(), f"N={N} K={K} M={M} G={G}")


@pytest.mark.parametrize("widths,K,M,G", [
    ((1024, 384), 4096, 72, 128),          # above 64 tokens, an odd slab inside
    ((512, 512, 512), 4096, 200, 64),
])
def test_several_matrices_and_the_folded_scale(widths, K, M, G):
    from paper_2306_00978_b200 import binding
    cases = [Case(6900 + i, n, K, M, G, 0.5) for i, n in enumerate(widths)]
    mats = [(*oracle_packed_to_cuda(c), c.N) for c in cases]
    x_raw = synth.activations(6990, M, K)
    inv_s = (np.float32(1.0) / cases[0].s).astype(np.float32)
    x = (x_raw.astype(np.float32) * inv_s[None, :]).astype(np.float16)
    plain = binding.linear_multi(to_cuda(x), mats, K, G)
    scaled = binding.linear_multi_scaled(to_cuda(x_raw), to_cuda(inv_s), mats, K, G)
    binding.poll_status()
    for c, y, ys in zip(cases, plain, scaled):
        assert_parity(y.cpu().numpy(), orc.linear(x, orc.dequantize(c.codes, c.zeros, c.scales, G)), f"N={c.N} of {widths}")
        assert np.array_equal(y.cpu().numpy().view(np.uint16), ys.cpu().numpy().view(np.uint16))


@pytest.mark.parametrize("N,K,M,G", [(4096, 4096, 100, 128), (1152, 8192, 130, 64), (640, 8192, 256, 128)])
def test_prefill_kernels_by_name_where_the_automatic_path_is_this_one(N, K, M, G):
    """AWQ_PATH_GEMM is the prefill kernels whatever awq_linear takes, and a name for this kernel ends at 64 tokens."""
    from paper_2306_00978_b200 import binding
    case = Case(6950 + N + K + M + G, N, K, M, G, 0.5)
    x, packed = to_cuda(case.x), oracle_packed_to_cuda(case)
    got = []
    for path in (binding.PATH_AUTO, binding.PATH_GEMM):
        binding.linear(x, *packed, N, K, G, path=path)
        n0 = binding.launch_count()
        y = binding.linear(x, *packed, N, K, G, path=path)
        got.append(binding.launch_count() - n0)
        assert_parity(y.cpu().numpy(), case.y_ref(), f"path {path}, N={N} K={K} M={M} G={G}")
    binding.poll_status()
    assert got == [2, 1]
    with pytest.raises(binding.AwqError):
        binding.linear(x, *packed, N, K, G, path=binding.PATH_GEMM_SKINNY)


def test_one_matrix_scaled_above_64_tokens_is_the_plain_call():
    from paper_2306_00978_b200 import binding
    N, K, M, G = 1024, 4096, 100, 128
    case = Case(6990, N, K, M, G, 0.5)
    packed = oracle_packed_to_cuda(case)
    x_raw = synth.activations(6991, M, K)
    inv_s = (np.float32(1.0) / case.s).astype(np.float32)
    x = (x_raw.astype(np.float32) * inv_s[None, :]).astype(np.float16)
    plain = binding.linear(to_cuda(x), *packed, N, K, G)
    scaled = binding.linear_multi_scaled(to_cuda(x_raw), to_cuda(inv_s), [(*packed, N)], K, G)[0]
    binding.poll_status()
    assert np.array_equal(plain.cpu().numpy().view(np.uint16), scaled.cpu().numpy().view(np.uint16))
