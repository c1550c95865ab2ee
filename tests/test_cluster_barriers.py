"""The kernels that run on clusters of two blocks, as text: an arrival that comes after its block's end cannot be made to show on a GPU."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_00978_b200", "csrc")


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu") and "cluster_wait()" in open(os.path.join(CSRC, f)).read())


def test_the_cluster_kernels_are_found():
    assert _sources() == ["gemm_stream.cu", "gemm_tcgen05_pair.cu"]


@pytest.mark.parametrize("source", ["gemm_stream.cu", "gemm_tcgen05_pair.cu"])
def test_a_block_outlives_the_other_blocks_arrivals(source):
    """A block may end, and its shared memory be given away, only when no arrival of the other block is on its way there: the
    warp that issues the products waits for the accumulators' last arrivals too, and where a block gives up the barrier in
    front of its end releases them.  Relaxed arrivals without either only at the start of a kernel."""
    text = open(os.path.join(CSRC, source)).read()
    kernel = text[text.index("__global__"):]
    start = kernel.index("griddepcontrol.launch_dependents")
    end = kernel.rindex("__syncthreads();", 0, kernel.index("tcgen05.dealloc"))
    assert "cluster_arrive_start();" in kernel[:start]
    assert "cluster_arrive_start();" not in kernel[start:]
    assert re.match(r"__syncthreads\(\);\s+cluster_sync_end\(\*ctl\.abort != 0u\);", kernel[end:])
    products = kernel[kernel.rindex("umma_pair_f16_a_tmem("):]
    products = products[:products.index("} else if (warp >= 8")]
    assert re.search(r"b < NACC && mbar_wait_warp\(acc_empty\(acc\), acc_phase \^ 1u, ctl\)", products)
    assert "barrier.cluster" not in text                    # the wrappers are the only spelling
    shared = open(os.path.join(CSRC, "tcgen05.cuh")).read()
    body = shared[shared.index("void cluster_sync_end("):]
    assert body.index("if (gave_up)") < body.index("barrier.cluster.arrive.release") < body.index("else") < body.index("cluster_wait()")
