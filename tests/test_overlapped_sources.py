"""Kernels that start while the kernel before them runs must not promise the compiler that what that kernel writes is constant: no
__restrict__ and no __ldg on the buffers that the calls hand from one kernel to the next."""
import os
import re

from paper_2410_13276_b200 import build

HANDED_ON = r"(?:scores|stats|row_ptr\w*|col_idx\w*|gq|gk|lse|src)"


def test_buffers_between_kernels_are_not_promised_constant():
    for name in ("gate_scores.cu", "mask.cu", "attn_tc.cu", "attn_tc_common.cuh"):
        text = re.sub(r"//[^\n]*", "", open(os.path.join(build.CSRC, name)).read())
        assert not re.findall(r"__restrict__\s+" + HANDED_ON + r"\b", text), name
        assert not re.findall(r"__ldg\([^;]*\b" + HANDED_ON + r"\b", text), name
