"""The binding's native call paths: the ordinary call and the Python path behind it give the same results
and refuse the same arguments."""
import numpy as np
import pytest

from tests.util import Case, oracle_packed_to_cuda, to_cuda


def test_tensors_on_the_host_are_refused():
    import torch
    from paper_2306_00978_b200 import binding
    binding.lib()
    x, b = torch.zeros((1, 128), dtype=torch.float16), torch.zeros(128 * 64, dtype=torch.uint8)
    assert binding._native.linear(x, b, x, b, 128, 128, 128, None, 0) is None
    assert binding._native.linear_int3(x, b, x, b, 128, 128, 128, None) is None


@pytest.mark.gpu
@pytest.mark.parametrize("N,K,M", [(128, 128, 1), (2048, 1152, 2), (256, 640, 33), (512, 512, 200)])
def test_same_as_the_python_path(N, K, M):
    import torch
    from paper_2306_00978_b200 import binding
    case = Case(600 + N + M, N, K, M, 128, 0.5)
    qw, sc, zp = oracle_packed_to_cuda(case)
    x = to_cuda(case.x)
    binding.linear(x, qw, sc, zp, N, K, np.int64(128))                       # an integer of another type: Python path
    out = torch.empty((M, N), dtype=torch.float16, device="cuda")
    assert binding._native.linear(x, qw, sc, zp, N, K, 128, out, 0) is out   # workspace is registered by now
    want = binding.linear(x, qw, sc, zp, N, K, np.int64(128))
    assert torch.equal(out, want) and torch.equal(binding.linear(x, qw, sc, zp, N, K, 128), want)
    q3 = binding.pack_int3(qw & 0x77, N, K)
    assert torch.equal(binding.linear_int3(x, q3, sc, zp, N, K, 128),
                       binding.linear_int3(x, q3, sc, zp, N, K, np.int64(128)))
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        side.wait_stream(torch.cuda.default_stream())
        y = binding.linear(x, qw, sc, zp, N, K, 128)
    side.synchronize()
    assert torch.equal(y, want)
    for bad in ((x.float(), qw, sc, zp, N, K, 128), (x, qw, sc.view(torch.int16), zp, N, K, 128),
                (x, qw, sc, zp, N, K + 128, 128), (x.t(), qw, sc, zp, N, K, 128), (x, qw, sc, zp, N, K, 100),
                (x, qw, sc, zp, N + 64, K, 128), (x[:, 1:], qw, sc, zp, N, K - 1, 128)):
        with pytest.raises(binding.AwqError):
            binding.linear(*bad)
    binding.poll_status()


@pytest.mark.gpu
def test_tensors_without_memory_raise():
    """A function transform passes wrappers without memory of their own; asking for an address throws in C++,
    which has to arrive as a Python exception from both calls."""
    import torch
    from paper_2306_00978_b200 import binding
    case = Case(640, 256, 256, 3, 128, 0.5)
    qw, sc, zp = oracle_packed_to_cuda(case)
    x = to_cuda(case.x)
    want = binding.linear(x, qw, sc, zp, 256, 256, 128)                      # registers the workspace
    q3 = binding.pack_int3(qw & 0x77, 256, 256)
    batch = torch.stack((x, x))
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda t: binding.linear(t, qw, sc, zp, 256, 256, 128))(batch)
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda t: binding.linear_int3(t, q3, sc, zp, 256, 256, 128))(batch)
    assert torch.equal(binding.linear(x, qw, sc, zp, 256, 256, 128), want)
    binding.poll_status()
