"""awq_linear with 2 to 8 tokens on long rows: where rows are at least 5/4 as long as the outputs are many, and up to 2^28 weights, the
stream kernel, else the chunked one (and the band kernel without a workspace)."""
import pytest

pytestmark = pytest.mark.gpu


def _operands(N, K, M, G, seed):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(seed)
    qw = torch.randint(0, 256, (N * K // 2,), dtype=torch.uint8, device="cuda", generator=gen)
    sc = (torch.rand((N // 16, K // G, 16), device="cuda", generator=gen) * 0.01 + 0.001).half()
    zp = torch.randint(0, 256, (N // 32, K // G, 16), dtype=torch.uint8, device="cuda", generator=gen)
    return qw, sc, zp, torch.randn((M, K), device="cuda", generator=gen).half()


@pytest.mark.parametrize("N,K,M,G,stream", [
    (8192, 10240, 3, 128, True), (8192, 10112, 3, 128, False),       # rows of 5/4 of the outputs
    (5504, 12288, 2, 64, True), (9856, 12288, 2, 64, False),
    (4096, 8192, 5, 128, True), (8192, 32768, 8, 128, True),         # the least and the most weights
    (8192, 32896, 8, 128, False),
])
def test_kernel_and_result(N, K, M, G, stream):
    import torch
    from paper_2306_00978_b200 import binding
    qw, sc, zp, x = _operands(N, K, M, G, N + K + M)
    auto = binding.linear(x, qw, sc, zp, N, K, G)
    assert torch.equal(auto, binding.linear(x, qw, sc, zp, N, K, G))
    # (asked for by name it is the chunked kernel on either side of the line)
    assert torch.equal(auto, binding.linear(x, qw, sc, zp, N, K, G, path=binding.PATH_GEMV_MID)) != stream
    assert not torch.equal(auto, binding.linear(x, qw, sc, zp, N, K, G, path=binding.PATH_GEMV))
    assert torch.equal(auto, binding.linear(x, qw, sc, zp, N, K, G, path=binding.PATH_GEMM_SKINNY)) == stream
    codes, scales, zeros = binding.unpack_canonical(qw, sc, zp, N, K, G)
    binding.poll_status()
    # sums in fp32 and one rounding to fp16: at most 2^-11 of a value, in the 2-norm below that
    err = ref = 0.0
    for n in range(0, N, 1024):
        rows = slice(n, min(n + 1024, N))
        diff = codes[rows].to(torch.float64).view(-1, K // G, G) - zeros[rows].to(torch.float64)[:, :, None]
        w = (diff * scales[rows].view(torch.float16).to(torch.float64)[:, :, None]).view(-1, K)
        want = x.double() @ w.t()
        err += float((auto[:, rows].double() - want).square().sum())
        ref += float(want.square().sum())
    assert (err / ref) ** 0.5 < 2.0 ** -11
