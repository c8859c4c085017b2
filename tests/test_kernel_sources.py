"""What a kernel's source must not hold, where no run shows it."""
import os
import re

import pytest

import paper_2510_19875_b200

CSRC = os.path.join(os.path.dirname(paper_2510_19875_b200.__file__), "csrc")
DEPENDENT = sorted(f for f in os.listdir(CSRC) if f.endswith(".cu") and "launch_kernel(" in open(os.path.join(CSRC, f)).read())


def code(name):
    return re.sub(r"//.*", "", open(os.path.join(CSRC, name)).read())


def test_the_kernels_are_found():
    assert DEPENDENT == ["attn_generic.cu", "attn_mma.cu", "attn_tc.cu", "attn_tok.cu", "mask_generic.cu", "mask_tc.cu", "mask_tok.cu"]


@pytest.mark.parametrize("name", DEPENDENT + ["common.cuh", "tc_common.cuh", "warp_common.cuh"])
def test_kernels_that_begin_early_read_no_memory_as_constant(name):
    """A programmatic dependent is alive while the kernel before it still writes. Read-only loads (__ldg, or inputs that are
    const and __restrict__) promise that nobody writes the data during the kernel's life."""
    text = code(name)
    assert not re.findall(r"__ldg\s*\(|ld\.global\.nc", text)
    assert not re.findall(r"const [\w: ]+\*\s*__restrict__", text)
