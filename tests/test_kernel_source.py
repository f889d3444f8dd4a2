"""Kernels launched programmatically are on the chip while the kernel before
them still writes: nothing they read from global memory may be promised to
the compiler as constant for the whole grid."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_05683_gb300", "csrc")


def test_no_read_only_promise_where_launches_are_programmatic():
    seen = 0
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        if "launch_pdl(" not in text:
            continue
        seen += 1
        code = re.sub(r"//[^\n]*", "", text)
        assert not re.search(r"__restrict__|__ldg\b|ld\.global\.nc", code), f
    assert seen
