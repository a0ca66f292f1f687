"""Kernels that stand on the SMs while the launch before them still runs: only data that was complete when they could start may be
read through the read-only path (__ldg), whose loads the compiler may move above the dependency wait."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_15806_b200", "csrc")

# what may be read that way, by file: the expanded layer (the row counts `cum`, the channel-block tables, the row scales) in the
# forward kernels, the weights and the level storage in the expansion; the explicit lowering is an ordinary launch
ALLOWED = {
    "pipe_expand.cu": {"src", "src + w", "reinterpret_cast<const uint4*>(row + kb * kStepBytes)", "reinterpret_cast<const uint2*>(row + kb * kStepBytes)",
                       "reinterpret_cast<const uint32_t*>(row + kb * kStepBytes)"},
    "pipe_quantize.cu": {"reinterpret_cast<const uint4*>(src)", "src + c"},   # lower_conv_input_kernel
    "pipe_gemm_direct.cu": {"cum + O / g", "cum + j", "cum + j + 1", "src", "src + 1"},
    "pipe_gemm_stream.cu": {"cum + O / g", "cum + j", "cum + j + 1", "p.f.order[br.k_begin + ko].scales + row0 + r"},
    "pipe_gemm_tc2.cu": {"br.blk + 1 + t.cb", "br.blk + 2 + t.cb", "cum + j0", "cum + j1", "p.f.branch[m].blk"},
    "pipe_common.cuh": {"cum + O / g", "cum + j", "cum + j + 1"},
}


def _arguments(text):
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__ldg\(", text):
        depth, i = 1, m.end()
        while depth:
            depth += {"(": 1, ")": -1}.get(text[i], 0)
            i += 1
        yield text[m.end():i - 1]


def test_every_file_whose_kernels_start_early_is_looked_at():
    early = set()
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            text = open(os.path.join(CSRC, name)).read()
            if "grid_wait(" in text or "griddepcontrol.wait" in text:
                early.add(name)
    assert early == set(ALLOWED)


@pytest.mark.parametrize("name", sorted(ALLOWED))
def test_the_read_only_path_reads_settled_data_only(name):
    for arg in _arguments(open(os.path.join(CSRC, name)).read()):
        assert arg in ALLOWED[name], arg
