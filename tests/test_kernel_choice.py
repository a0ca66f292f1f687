"""The diagnostic selector: every number forces one kernel alone, so that a test which names a kernel reaches it."""
import os
import re

from paper_2311_15806_b200 import binding as B

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_every_number_of_the_selector_forces_one_kernel():
    text = open(os.path.join(ROOT, "paper_2311_15806_b200", "csrc", "pipe_forward.cu")).read()
    text = text[text.index("static pipe_status dispatch_forward(const ForwardArgs& a", text.index("static pipe_status run_forward")):]
    text = text[text.index("return PIPE_ERR_UNSUPPORTED;"):text.index('extern "C"')]   # (behind the branch for zero points)
    forced = dict(re.findall(r"if \(choice == (\d)\) return (forward_\w+)\(", text))
    assert {int(k): v for k, v in forced.items()} == {
        B.KERNEL_REFERENCE: "forward_reference", B.KERNEL_TCGEN05: "forward_tcgen05", B.KERNEL_STREAM: "forward_stream",
        B.KERNEL_TCGEN05_PAIR: "forward_tcgen05_pair", B.KERNEL_DECODE_TC: "forward_decode_tc", B.KERNEL_DIRECT: "forward_direct"}
    assert len(re.findall(r"choice == \d", text)) == 6


def test_the_selector_takes_every_kernel_and_nothing_else():
    lib = B.lib()
    try:
        for which in range(B.KERNEL_DIRECT + 1):
            assert lib.pipe_diag_select_kernel(which) == B.PIPE_OK
        for which in (-1, B.KERNEL_DIRECT + 1):
            assert lib.pipe_diag_select_kernel(which) == B.PIPE_ERR_INVALID_ARG
    finally:
        lib.pipe_diag_select_kernel(B.KERNEL_AUTO)
