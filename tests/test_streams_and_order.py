"""Calls on several streams and threads: those that need no workspace may overlap."""
import threading

import numpy as np
import pytest

from tests.util import Case, oracle_packed_to_cuda, to_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("widths,K,M,G", [((4096, 2304), 5248, 4, 128), ((2176, 4352), 8192, 8, 64)])
def test_several_matrices_up_to_8_tokens_need_no_workspace(widths, K, M, G):
    """Long rows, many output rows: one launch of the band kernel, bit for bit what it gives each matrix alone, and nothing that two
    streams or threads would share."""
    import torch
    from paper_2306_00978_b200 import binding
    cases = [Case(6900 + i, n, K, M, G, 0.5) for i, n in enumerate(widths)]
    mats = [(*oracle_packed_to_cuda(c), c.N) for c in cases]
    inv_s = to_cuda((np.float32(1.0) / cases[0].s).astype(np.float32))
    xs = [torch.randn((M, K), device="cuda").half() for _ in range(2)]
    scaled_x = [(x.float() * inv_s).half() for x in xs]
    want = [[binding.linear(x, *m[:3], m[3], K, G, path=binding.PATH_GEMV) for m in mats] for x in xs]
    want_scaled = [[binding.linear(x, *m[:3], m[3], K, G, path=binding.PATH_GEMV) for m in mats] for x in scaled_x]
    n0 = binding.launch_count()
    plain = binding.linear_multi(xs[0], mats, K, G)
    assert binding.launch_count() - n0 == 1
    assert all(torch.equal(y, w) for y, w in zip(plain, want[0]))
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream() for _ in xs]
    got = [[], []]

    def calls(i):
        with torch.cuda.stream(streams[i]):
            for _ in range(40):
                got[i].append((binding.linear_multi(xs[i], mats, K, G), binding.linear_multi_scaled(xs[i], inv_s, mats, K, G)))

    threads = [threading.Thread(target=calls, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    binding.poll_status()
    for i in range(2):
        assert len(got[i]) == 40
        for plain, scaled in got[i]:
            assert all(torch.equal(y, w) for y, w in zip(plain, want[i]))
            assert all(torch.equal(y, w) for y, w in zip(scaled, want_scaled[i]))
