"""Kernels that are resident while the kernel in front writes what they read, as text: a stale line of the read-only path cannot be made to
show on a GPU.  They read global memory through L2."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_00978_b200", "csrc")


def _kernels():
    found = {}
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith(".cu"):
            continue
        text = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"__global__[^{;]*?(\w+_kernel)\s*\(([^{]*)\)\s*\{", text):
            body = text[m.end():text.index("\n}\n", m.end())]
            if "start_behind_predecessor();" in body:
                found[m.group(1)] = (m.group(2), body)
    return found


def test_the_kernels_are_found():
    assert sorted(_kernels()) == ["channel_scales_kernel", "clip_search_kernel", "quantize_pack_tile_kernel", "sqdiff_final_kernel"]


@pytest.mark.parametrize("name", ["channel_scales_kernel", "clip_search_kernel", "quantize_pack_tile_kernel", "sqdiff_final_kernel"])
def test_nothing_is_read_as_read_only_data(name):
    parameters, body = _kernels()[name]
    assert "__ldg(" not in body and ".nc" not in body
    inputs = re.findall(r"const (?:float|double|__half)\*\s*(__restrict__)?\s*(\w+)", parameters)
    assert inputs and not any(restrict for restrict, _ in inputs)
    for _, pointer in inputs:                            # every other use is an address
        assert not re.search(rf"\b{pointer}\[", body), pointer
