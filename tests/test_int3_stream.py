"""awq_linear_int3 where the stream kernel serves awq_linear: it reads the 3-bit storage, without an expansion, and gives the bits of
awq_linear on the expanded array (the same kernel on the same codes, which the other tests hold against the oracle)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,K,M,G", [
    (128, 128, 9, 128),        # half a tile of channels, half a stage
    (1024, 1408, 16, 64),      # a last stage of two k-blocks
    (2176, 2304, 17, 128),     # an odd slab, the 32-token form
    (384, 8192, 32, 64),       # tiles cut over many pairs
    (4096, 4224, 33, 128),     # scales in the product from 33 tokens
    (11008, 4096, 64, 128),
    (1024, 4096, 3, 256),      # few output rows: this kernel below 9 tokens too; a group's entry twice
])
def test_same_bits_as_on_the_expanded_array(N, K, M, G):
    import torch
    from paper_2306_00978_b200 import binding
    gen = torch.Generator(device="cuda").manual_seed(N + K + M)
    stored = min(G, 128)
    qw3 = torch.randint(0, 256, (N * K // 8 * 3,), dtype=torch.uint8, device="cuda", generator=gen)
    sc = (torch.rand((N // 16, K // stored, 16), device="cuda", generator=gen) * 0.01 + 0.001).half()
    zp = (torch.randint(0, 256, (N // 32, K // stored, 16), dtype=torch.uint8, device="cuda", generator=gen) & 0x77)
    x = torch.randn((M, K), device="cuda", generator=gen).half()
    qw = torch.empty(N * K // 2, dtype=torch.uint8, device="cuda")
    assert binding.lib().awq_unpack_int3(qw3.data_ptr(), qw.data_ptr(), N, K, torch.cuda.current_stream().cuda_stream) == 0
    scratch = torch.full((N * K // 2,), 0xA5, dtype=torch.uint8, device="cuda")
    want = binding.linear(x, qw, sc, zp, N, K, G)
    got = binding.linear_int3(x, qw3, sc, zp, N, K, G, scratch=scratch)
    alone = binding.linear_int3(x, qw3, sc, zp, N, K, G)
    binding.poll_status()
    assert torch.equal(got, want) and torch.equal(alone, want)
    assert bool((scratch == 0xA5).all())                 # nothing was expanded


def test_scratch_only_where_the_storage_is_expanded():
    import numpy as np
    import torch
    from paper_2306_00978_b200 import binding
    N, K, G = 2048, 2048, 128
    L = binding.lib()
    qw3 = torch.randint(0, 256, (N * K // 8 * 3,), dtype=torch.uint8, device="cuda")
    sc, zp = torch.rand((N // 16, K // G, 16), device="cuda").half(), torch.zeros((N // 32, K // G, 16), dtype=torch.uint8, device="cuda")
    scratch = torch.empty(N * K // 2, dtype=torch.uint8, device="cuda")

    def call(M, given):
        x, y = torch.ones((M, K), device="cuda").half(), torch.empty((M, N), dtype=torch.float16, device="cuda")
        n0 = binding.launch_count()
        rc = L.awq_linear_int3(x.data_ptr(), qw3.data_ptr(), sc.data_ptr(), zp.data_ptr(), y.data_ptr(),
                               scratch.data_ptr() if given else None, M, N, K, G, torch.cuda.current_stream().cuda_stream)
        assert rc == 0 or binding.launch_count() == n0
        return rc

    for M in (8, 9, 64, 65):
        binding.ensure_workspace(binding.workspace_bytes(M, N, K, G))
    ws = binding._workspace[torch.cuda.current_device()]
    assert [call(M, False) for M in (8, 9, 64, 65)] == [0, 0, 0, 1]
    for M, more in ((9, False), (64, False), (65, True)):
        for group in (G, np.int64(G)):                       # the native call and the one through ctypes
            x = torch.ones((M, K), device="cuda").half()
            torch.cuda.synchronize()
            torch.cuda.reset_peak_memory_stats()
            before = torch.cuda.memory_allocated()
            binding.linear_int3(x, qw3, sc, zp, N, K, group)
            assert (torch.cuda.max_memory_allocated() - before >= N * K // 2) == more
    binding.poll_status()
    try:                                                     # without a workspace for its parts the stream kernel is not taken
        assert L.awq_set_workspace(None, 0) == 0
        assert call(9, False) == 1 and call(9, True) == 0
        binding.poll_status()
    finally:
        assert L.awq_set_workspace(ws.data_ptr(), ws.numel()) == 0
