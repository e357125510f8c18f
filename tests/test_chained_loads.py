"""Kernels that start before the one ahead of them has ended (launch_chained)
read global memory with plain loads only: a read-only load (__ldg, ld.global.nc)
says that the value is constant for the kernel's life, so it may be moved above
the wait for the kernel ahead, whose results (C, dC, activations) it would then
miss."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_26430_gb300", "csrc")


def source(f):
    txt = open(os.path.join(CSRC, f)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", txt, flags=re.S)


# the contraction path's kernels are launched plainly: after all work ahead
CHAINED = sorted(f for f in os.listdir(CSRC) if f.endswith(".cuh") and f != "framefb_dense.cuh")


def test_the_contraction_path_is_not_chained():
    assert "chain_wait" not in source("framefb_dense.cuh") and "launch_chained" not in source("framefb_dense.cu")


@pytest.mark.parametrize("f", CHAINED)
def test_no_read_only_loads(f):
    assert not re.findall(r"__ldg\s*\(|\.global\.nc\b", source(f))


@pytest.mark.parametrize("f", CHAINED)
def test_every_kernel_waits_first(f):
    """The first statement of every kernel of these files is the wait."""
    heads = re.findall(r"__global__[^;{]*?\)\s*\{\s*([^\n]*)", source(f))
    assert all(h.strip() == "chain_wait();" for h in heads), heads
