"""The binding's workspace: what a stream capture may and may not do, and that a call's result does not depend
on which calls came before it."""
import numpy as np
import pytest

from tests.util import Case, assert_parity, oracle_packed_to_cuda, to_cuda


def test_nothing_is_registered_while_capturing(monkeypatch):
    import torch
    from paper_2306_00978_b200 import binding

    def not_now(*a, **k):
        raise AssertionError("allocated, registered or synchronized while capturing")
    monkeypatch.setattr(binding, "_workspace", {})
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: True)
    monkeypatch.setattr(torch.cuda, "synchronize", not_now)
    monkeypatch.setattr(torch, "empty", not_now)
    binding.ensure_workspace(1 << 20)
    assert not binding._workspace


def test_replaced_workspaces_stay_alive_and_bounded(monkeypatch):
    """A graph holds the address of the workspace it was captured with, so growing must not free it."""
    import torch
    import weakref
    from paper_2306_00978_b200 import binding

    class Library:
        def awq_set_workspace(self, address, nbytes):
            return 0
    real = torch.empty
    monkeypatch.setattr(binding, "_workspace", {})
    monkeypatch.setattr(binding, "_replaced", [], raising=False)
    monkeypatch.setattr(binding, "lib", Library)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "is_current_stream_capturing", lambda: False)
    monkeypatch.setattr(torch.cuda, "synchronize", lambda: None)
    monkeypatch.setattr(torch, "empty", lambda n, dtype, device: real(n, dtype=dtype))
    seen = []
    for need in (1 << 10, (1 << 22) + 1, (1 << 22) + 2, 9 << 20, 10 << 20, 40 << 20):
        binding.ensure_workspace(need)
        buf = binding._workspace[0]
        assert buf.numel() >= need
        if not seen or seen[-1]() is not buf:
            seen.append(weakref.ref(buf))
        del buf
    assert len(seen) > 2 and all(r() is not None for r in seen)
    assert sum(r().numel() for r in seen[:-1]) < binding._workspace[0].numel()


class _NoWorkspace:
    """Nothing registered inside, what was registered is registered again afterwards."""

    def __enter__(self):
        import torch
        from paper_2306_00978_b200 import binding
        torch.cuda.synchronize()
        self.dev = torch.cuda.current_device()
        self.saved = binding._workspace.pop(self.dev, None)
        assert binding.lib().awq_set_workspace(None, 0) == 0

    def __exit__(self, *exc):
        import torch
        from paper_2306_00978_b200 import binding
        torch.cuda.synchronize()
        binding._workspace.pop(self.dev, None)
        assert binding.lib().awq_set_workspace(None, 0) == 0
        if self.saved is not None:
            assert binding.lib().awq_set_workspace(self.saved.data_ptr(), self.saved.numel()) == 0
            binding._workspace[self.dev] = self.saved


@pytest.mark.gpu
@pytest.mark.parametrize("M", [32, 48, 200])
def test_several_matrices_in_a_capture(M):
    """linear_multi in a capture: without a call before it the kernels that need no workspace, after one the
    bits of the call outside."""
    import torch
    from paper_2306_00978_b200 import binding
    K, G = 1408, 128
    cases = [Case(9300 + i, n, K, M, G, 0.5) for i, n in enumerate((384, 256))]
    mats = [(*oracle_packed_to_cuda(c), c.N) for c in cases]
    x = to_cuda(cases[0].x)
    outs = [torch.zeros((M, c.N), dtype=torch.float16, device="cuda") for c in cases]

    def captured():
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            binding.linear_multi(x, mats, K, G, outs=outs)
        graph.replay()
        binding.poll_status()
        return [y.clone() for y in outs]

    with _NoWorkspace():
        binding.poll_status()
        for y, c in zip(captured(), cases):
            assert not binding._workspace
            c.x = cases[0].x
            assert_parity(y.cpu().numpy(), c.y_ref(), f"captured without a workspace, M={M}, N={c.N}")
        eager = binding.linear_multi(x, mats, K, G)
        for y, want in zip(captured(), eager):
            assert torch.equal(y, want)


@pytest.mark.gpu
@pytest.mark.parametrize("N,K,M,multi", [
    (1152, 8192, 130, False),     # 9 slabs: ten tiles on the stream kernel, which only runs with a workspace
    (1152, 8192, 130, True),
    (1152, 8192, 300, False),     # 25 half-empty tiles, balanced over the SM pairs by stream-K
    (1024, 8192, 300, True),
])
def test_same_bits_before_and_after_a_larger_call(N, K, M, multi):
    import torch
    from paper_2306_00978_b200 import binding
    G = 128
    torch.manual_seed(N + M)
    qw = torch.randint(0, 256, (N * K // 2,), dtype=torch.uint8, device="cuda")
    sc = (torch.rand((N // 16, K // G, 16), device="cuda") * 0.01 + 0.001).half()
    zp = torch.randint(0, 256, (N // 32, K // G, 16), dtype=torch.uint8, device="cuda")
    x = torch.randn((M, K), device="cuda").half()

    def call():
        return binding.linear_multi(x, [(qw, sc, zp, N)], K, G)[0] if multi else binding.linear(x, qw, sc, zp, N, K, G)

    with _NoWorkspace():
        first = call()
        binding.ensure_workspace(1 << 28)
        second = call()
        binding.poll_status()
        assert torch.equal(first, second)


@pytest.mark.gpu
def test_a_workspace_is_no_slower_than_none():
    """130 tokens on 28672 -> 1152: ten tiles for all SM pairs.  With room for the partial sums of no tile width
    the tile is the one that is best without them (not the one that would have been best with them); with
    room for them a tile is not cut among so many pairs that adding their sums costs more than it saves."""
    import torch
    from paper_2306_00978_b200 import binding
    N, K, M, G = 1152, 28672, 130, 128
    qw = torch.randint(0, 256, (N * K // 2,), dtype=torch.uint8, device="cuda")
    sc = (torch.rand((N // 16, K // G, 16), device="cuda") * 0.01 + 0.001).half()
    zp = torch.randint(0, 256, (N // 32, K // G, 16), dtype=torch.uint8, device="cuda")
    x = torch.randn((M, K), device="cuda").half()
    y = torch.empty((M, N), dtype=torch.float16, device="cuda")
    L, us = binding.lib(), {}

    def call():
        assert L.awq_linear(x.data_ptr(), qw.data_ptr(), sc.data_ptr(), zp.data_ptr(), y.data_ptr(), M, N, K, G, None) == 0

    with _NoWorkspace():
        for nbytes in (0, 1 << 22, 5 << 20, 20 << 20):       # none, too small, one for 64-token tiles, one for all
            buf = torch.empty(max(nbytes, 1), dtype=torch.uint8, device="cuda")
            assert L.awq_set_workspace(buf.data_ptr() if nbytes else None, nbytes) == 0
            best = float("inf")
            for _ in range(20):
                begin, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
                begin.record()
                for _ in range(4):
                    call()
                end.record()
                end.synchronize()
                best = min(best, begin.elapsed_time(end) * 250.0)
            us[nbytes] = best
            binding.poll_status()
            assert L.awq_set_workspace(None, 0) == 0
    assert us[1 << 22] < 1.25 * us[0] and us[5 << 20] < us[0] and us[20 << 20] < us[0], us
