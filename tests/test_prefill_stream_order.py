"""The SM-pair prefill kernel and the stream kernel copy packed weights before the work in front of them in the stream has completed:
calls right behind the library's own writers, and chains of calls that read what the one before wrote, give what they give alone."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M,bits", [
    (2048, 2048, 300, 4),       # 128-token tiles
    (1024, 4096, 1000, 4),      # 256-token tiles
    (4096, 4096, 700, 3),       # behind the kernel that expands the 3-bit storage
    (4096, 4096, 16, 3),        # behind the kernel that packs it: the stream kernel reads it as it is
    (2048, 4096, 48, 3),
    (4096, 4096, 16, 4),        # behind the quantizer
])
def test_calls_behind_the_writers_of_their_operands(N, K, M, bits):
    import torch
    from paper_2306_00978_b200 import binding
    G = 128
    torch.manual_seed(N + M)
    W = [(torch.randn(N, K, device="cuda") * 0.02).half() for _ in range(3)]
    stat = torch.rand(K, device="cuda") + 0.5
    x = torch.randn(M, K, device="cuda").half()

    def layer(w, x):
        qw, sc, zp = binding.quantize_pack(w, stat, 0.5, G, bits=bits)
        if bits == 3:
            return binding.linear_int3(x, binding.pack_int3(qw, N, K), sc, zp, N, K, G)
        return binding.linear(x, qw, sc, zp, N, K, G)

    want = []
    for w in W:
        torch.cuda.synchronize()
        want.append(layer(w, x))
        torch.cuda.synchronize()
    for it in range(20):
        for y, w in zip([layer(w, x) for w in W], want):
            assert torch.equal(y, w), it
    binding.poll_status()


def test_a_chain_of_square_layers():
    import torch
    from paper_2306_00978_b200 import binding
    N, M, G = 2048, 500, 128
    torch.manual_seed(5)
    stat = torch.rand(N, device="cuda") + 0.5
    packed = [binding.quantize_pack((torch.randn(N, N, device="cuda") * 0.02).half(), stat, 0.0, G) for _ in range(4)]
    x = torch.randn(M, N, device="cuda").half()

    def chain(sync):
        h = x
        for p in packed:
            h = binding.linear(h, *p, N, N, G)
            if sync:
                torch.cuda.synchronize()
        return h

    want = chain(True)
    for _ in range(50):
        assert torch.equal(chain(False), want)
    binding.poll_status()
