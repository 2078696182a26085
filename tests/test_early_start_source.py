"""The CSR build's kernels may start while their predecessors still write: each
begins by waiting for them, and none reads the chain's buffers through the
read-only path, which is for data that stays as it is while a kernel is
resident."""
import os
import re

from paper_2502_08042_gb300 import _native

INPUTS = {"gv"}  # pointers no kernel of the chain writes


def source():
    with open(os.path.join(_native.CSRC, "csr_build.cu")) as f:
        return re.sub(r"//[^\n]*", "", f.read())


def test_every_kernel_waits_first():
    kernels = re.findall(r"__global__[^{;]*\{\s*([^;]*);", source())
    assert len(kernels) >= 8
    assert set(kernels) == {"wait_predecessor()"}


def test_no_read_only_loads_of_the_chains_buffers():
    text = source()
    assert "__ldg(" not in text and "ld.global.nc" not in text
    assert set(re.findall(r"__restrict__\s+(\w+)", text)) <= INPUTS
