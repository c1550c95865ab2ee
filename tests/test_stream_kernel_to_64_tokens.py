"""The stream kernel (awq_linear with 9 .. 64 tokens, and fewer where the output rows are few): token tiles, groups, short last
stages, tiles in few and in many parts, several matrices in one launch, against the fp64 oracle."""
import numpy as np
import pytest

from oracle import awq_oracle as orc
from paper_2306_00978_b200 import synth
from tests.util import Case, assert_parity, oracle_packed_to_cuda, to_cuda

pytestmark = pytest.mark.gpu


def unrounded_bound(x, W):
    """Up to 32 tokens nothing is rounded before the output: the products (q - z) * x are exact in the
    tensor core, their sums, the multiplications by Delta and the sums over groups and parts are fp32.
    At most K + 64 roundings of 2^-24 act on partial results bounded by sum |W||x|; the fp16 output adds
    2^-11 of the value (or 2^-25 in its subnormal range)."""
    a = np.abs(x.astype(np.float64)) @ np.abs(W).T
    ref = x.astype(np.float64) @ W.T
    return ref, 2.0 ** -11 * np.abs(ref) + 2.0 ** -25 + (x.shape[1] + 64) * 2.0 ** -24 * a


@pytest.mark.parametrize("N,K,M,G", [
    (128, 128, 1, 64), (128, 128, 9, 128),        # half a tile of half a stage; few rows: also below 9 tokens
    (256, 384, 16, 128),                           # two parts, the second of half a stage
    (384, 2176, 17, 64),                           # an odd slab, nine parts, 32-token tile
    (1152, 4224, 32, 128),                         # ranges of one and two stages, nine to seventeen parts
    (128, 9088, 8, 128),                           # half a tile in 36 parts
    (19072, 640, 12, 64),                          # 75 tiles of three stages for 74 pairs: ranges of three and four stages
    (2048, 5120, 31, 256),                         # a group stored per 128 columns
    (512, 1152, 33, 64), (1280, 3200, 64, 128),    # 48 and 64 tokens a tile
])
def test_linear(N, K, M, G):
    from paper_2306_00978_b200 import binding
    case = Case(7000 + N + K + M + G, N, K, M, G, 0.5)
    packed = oracle_packed_to_cuda(case)
    y = binding.linear(to_cuda(case.x), *packed, N, K, G)
    again = binding.linear(to_cuda(case.x), *packed, N, K, G)
    binding.poll_status()
    y = y.cpu().numpy()
    assert np.array_equal(y.view(np.uint16), again.cpu().numpy().view(np.uint16))
    if M <= 32:
        ref, bound = unrounded_bound(case.x, orc.dequantize(case.codes, case.zeros, case.scales, G))
        assert (np.abs(y.astype(np.float64) - ref) <= bound).all()
    else:
        assert_parity(y, case.y_ref(), f"N={N} K={K} M={M} G={G}")


@pytest.mark.parametrize("widths,K,M,G", [
    ((256, 128, 384), 1408, 10, 128),              # three matrices, slabs end to end, two of them odd
    ((1024, 1024), 4096, 32, 64),
    ((512, 128, 128, 896), 2688, 48, 128),
])
def test_several_matrices_and_the_folded_scale(widths, K, M, G):
    """One launch (and the kernel that adds the parts) serves all matrices; the scaled call gives bit for
    bit what the plain one gives on x' = fp16(x * inv_s)."""
    from paper_2306_00978_b200 import binding
    cases = [Case(8100 + i, n, K, M, G, 0.5) for i, n in enumerate(widths)]
    mats = [(*oracle_packed_to_cuda(c), c.N) for c in cases]
    x_raw = synth.activations(8199, M, K)
    inv_s = (np.float32(1.0) / cases[0].s).astype(np.float32)
    x = (x_raw.astype(np.float32) * inv_s[None, :]).astype(np.float16)
    plain = binding.linear_multi(to_cuda(x), mats, K, G)
    n0 = binding.launch_count()
    scaled = binding.linear_multi_scaled(to_cuda(x_raw), to_cuda(inv_s), mats, K, G)
    assert binding.launch_count() - n0 == 2
    binding.poll_status()
    for c, y, ys in zip(cases, plain, scaled):
        ref = orc.linear(x, orc.dequantize(c.codes, c.zeros, c.scales, G))
        assert_parity(y.cpu().numpy(), ref, f"N={c.N} of {widths}")
        assert np.array_equal(y.cpu().numpy().view(np.uint16), ys.cpu().numpy().view(np.uint16))


@pytest.mark.parametrize("N,K,M", [
    (8192, 4096, 24),              # ranges of six and seven stages, fewer than the ring's
    (8192, 4096, 32),
    (22016, 4096, 32),             # eighteen and nineteen stages: the ring wraps twice
])
def test_back_to_back_calls_on_new_operands(N, K, M):
    """Operands made on the device, two calls on them with nothing in between: equal bit for bit, and every
    eighth pair within the rounding bound of the product in fp64.  A stage of the weight ring that is refilled
    under a reader shows as wrong channels of one band in about one call out of 400 where the ring wraps early."""
    import torch
    from paper_2306_00978_b200 import binding
    G = 128
    torch.manual_seed(N + K + M)
    for it in range(400):
        qw = torch.randint(0, 256, (N * K // 2,), dtype=torch.uint8, device="cuda")
        sc = (torch.rand((N // 16, K // G, 16), device="cuda") * 0.01 + 0.001).half()
        zp = torch.randint(0, 256, (N // 32, K // G, 16), dtype=torch.uint8, device="cuda")
        x = torch.randn((M, K), device="cuda").half()
        y = binding.linear(x, qw, sc, zp, N, K, G)
        again = binding.linear(x, qw, sc, zp, N, K, G)
        binding.poll_status()
        differ = (y != again).nonzero()
        assert differ.numel() == 0, (it, differ.shape[0], sorted({int(n) // 16 for n in differ[:, 1]}))
        if it % 8 == 0:
            codes, s, z = binding.unpack_canonical(qw, sc, zp, N, K, G)
            W = (codes.view(N, K // G, G).double() - z.double()[:, :, None]).mul_(s.double()[:, :, None]).view(N, K)
            ref, a = x.double() @ W.T, x.double().abs() @ W.abs().T
            bound = 2.0 ** -11 * ref.abs() + 2.0 ** -25 + (K + 64) * 2.0 ** -24 * a    # as in unrounded_bound
            assert bool(((y.double() - ref).abs() <= bound).all()), it
