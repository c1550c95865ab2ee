"""The layer call's own output tensor, where it is allocated past the dispatcher and where something takes part in the allocation."""
import contextlib

import pytest


class _Calls:
    """A dispatch mode that lists what passes through it."""

    def __new__(cls, names):
        import torch
        from torch.utils._python_dispatch import TorchDispatchMode

        class Mode(TorchDispatchMode):
            def __torch_dispatch__(self, func, types, args=(), kwargs=None):
                names.append(str(func))
                return func(*args, **(kwargs or {}))
        return Mode()


@pytest.mark.gpu
@pytest.mark.parametrize("context", ["plain", "no_grad", "inference", "mode", "deterministic"])
def test_output(context):
    import torch
    from paper_2306_00978_b200 import binding
    N, K, M, G = 256, 512, 2, 128
    torch.manual_seed(5)
    W = (torch.randn(N, K, device="cuda") * 0.02).half()
    packed = binding.quantize_pack(W, None, 0.0, G)
    x = torch.randn(M, K, device="cuda").half()
    given = torch.empty(M, N, dtype=torch.float16, device="cuda")
    binding.linear(x, *packed, N, K, G, out=given)
    names = []
    before = torch.are_deterministic_algorithms_enabled()
    managers = {"plain": contextlib.nullcontext, "no_grad": torch.no_grad, "inference": torch.inference_mode, "mode": lambda: _Calls(names),
                "deterministic": contextlib.nullcontext}
    try:
        if context == "deterministic":
            torch.use_deterministic_algorithms(True)
        with managers[context]():
            y = binding.linear(x, *packed, N, K, G)
    finally:
        torch.use_deterministic_algorithms(before)
    assert y.shape == (M, N) and y.dtype == torch.float16 and y.device == x.device and y.is_contiguous() and not y.requires_grad
    assert torch.equal(y, given) and y.is_inference() == (context == "inference")
    assert any("empty" in n for n in names) == (context == "mode")
    other = binding.linear(x, *packed, N, K, G)
    assert other.data_ptr() != y.data_ptr() and (other + 1).sum().isfinite()
