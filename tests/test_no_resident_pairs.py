"""A device, or a partition of one, on which no pair of SMs can be had: awq_linear takes the kernels that need none.  The runtime's
answer is replaced by a shared object loaded in front of it, in a process of its own."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SHIM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdlib.h>
/* FAKE_PAIRS: "none": no cluster is ever resident; "fails once": the first query is answered with an error */
int cudaOccupancyMaxActiveClusters(int* n, const void* kernel, const void* config) {
    static int asked = 0;
    if (getenv("FAKE_PAIRS")[0] == 'n') { *n = 0; return 0; }
    if (asked++ == 0) return 999;
    return ((int (*)(int*, const void*, const void*))dlsym(RTLD_NEXT, "cudaOccupancyMaxActiveClusters"))(n, kernel, config);
}
"""

PROGRAM = """
import sys
import torch
from paper_2306_00978_b200 import binding, synth
from tests.util import Case, assert_parity, oracle_packed_to_cuda, to_cuda

def launches(call):
    n0 = binding.launch_count()
    y = call()
    binding.poll_status()
    return y, binding.launch_count() - n0

G = 128
if sys.argv[1] == "none":
    for N, K, M in ((256, 1024, 4), (1024, 4096, 16), (640, 1152, 48), (1024, 4096, 100), (512, 1024, 300)):
        case = Case(9100 + M, N, K, M, G, 0.5)
        packed, x = oracle_packed_to_cuda(case), to_cuda(case.x)
        for _ in range(2):
            y, n = launches(lambda: binding.linear(x, *packed, N, K, G))
            assert n == 1, (M, n)
            assert_parity(y.cpu().numpy(), case.y_ref(), f"M={M}")
        inv_s = to_cuda((1.0 / case.s).astype("float32"))
        both = binding.linear_multi(x, [(*packed, N)] * 2, K, G) + binding.linear_multi_scaled(x * 0, inv_s, [(*packed, N)] * 2, K, G)
        binding.poll_status()
        assert torch.equal(both[0], both[1]) and not both[2].any() and not both[3].any()
        assert_parity(both[0].cpu().numpy(), case.y_ref(), f"several, M={M}")
    N, K, M = 4096, 8320, 5                  # few tokens on long rows: the chunked kernel and the one that adds its parts
    qw = torch.randint(0, 256, (N * K // 2,), dtype=torch.uint8, device="cuda")
    sc, zp = torch.rand((N // 16, K // G, 16), device="cuda").half(), torch.randint(0, 256, (N // 32, K // G, 16), dtype=torch.uint8, device="cuda")
    long_x = torch.randn((M, K), device="cuda").half()
    binding.linear(long_x, qw, sc, zp, N, K, G)
    y, n = launches(lambda: binding.linear(long_x, qw, sc, zp, N, K, G))
    assert n == 2 and torch.equal(y, binding.linear(long_x, qw, sc, zp, N, K, G, path=binding.PATH_GEMV_MID))
    N, K, M = 2048, 1024, 16                 # 3-bit storage: expanded, and the prefill kernel behind it
    qw3 = torch.randint(0, 256, (N * K // 8 * 3,), dtype=torch.uint8, device="cuda")
    sc, zp = torch.rand((N // 16, K // G, 16), device="cuda").half(), torch.randint(0, 8, (N // 32, K // G, 16), dtype=torch.uint8, device="cuda")
    some_x = torch.randn((M, K), device="cuda").half()
    y, n = launches(lambda: binding.linear_int3(some_x, qw3, sc, zp, N, K, G))
    assert n == 2 and torch.equal(y, binding.linear(some_x, binding.unpack_int3(qw3, N, K), sc, zp, N, K, G))
    N, K = 512, 1024
    try:
        binding.linear(x[:16], *packed, N, K, G, path=binding.PATH_GEMM_SKINNY)
        raise SystemExit("a kernel asked for by name must not be replaced")
    except binding.AwqError:
        pass
else:
    N, K, M = 1024, 4096, 16
    case = Case(9200, N, K, M, G, 0.5)
    packed, x = oracle_packed_to_cuda(case), to_cuda(case.x)
    seen = []
    for _ in range(2):
        y, n = launches(lambda: binding.linear(x, *packed, N, K, G))
        seen.append(n)
        assert_parity(y.cpu().numpy(), case.y_ref(), "")
    assert seen == [1, 2], seen               # the prefill kernel, then the stream kernel with the one that adds its parts
print("done")
"""


@pytest.mark.parametrize("fake", ["none", "fails once"])
def test_the_automatic_path_without_pairs(fake, tmp_path):
    source, shim = tmp_path / "shim.c", tmp_path / "shim.so"
    source.write_text(SHIM)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(shim), str(source), "-ldl"], check=True)
    env = dict(os.environ, LD_PRELOAD=str(shim), FAKE_PAIRS=fake, PYTHONPATH=ROOT)
    done = subprocess.run([sys.executable, "-c", PROGRAM, fake], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert done.returncode == 0 and done.stdout.strip().endswith("done"), done.stdout + done.stderr
