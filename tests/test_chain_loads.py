"""Chained kernels (programmatic dependents) read what the kernels before them write with ordinary loads: the sources
of the network's kernels hold no read-only load of such data."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1503_01722_gb300", "csrc")
FILES = ["ocmc_unet.cu", "ocmc_unet_kernels.cuh", "ocmc_unet_tc.cu", "ocmc_unet_wgrad_tc.cu", "ocmc_umma.cuh"]
# the caller's maps and the network's weights are complete before a chain starts
CALLERS = {"dose", "dens", "sigma", "target", "w", "b"}


def source(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", FILES)
def test_read_only_loads(name):
    s = source(name)
    assert "__ldg" not in s and "ld.global.nc" not in s
    kernels = re.findall(r"__global__\s+void\s+(?:__launch_bounds__\([^)]*\)\s*)?(\w+)\s*\(([^{]*?)\)\s*\{(.*?)\n\}", s, re.S)
    chained = [k for k in kernels if "chain_wait()" in k[2]]
    assert len(chained) == s.count("chain_next()") and "__restrict__" not in "".join(re.findall(r"struct[^;{]*\{[^}]*\}", s))
    for kernel, args, _ in chained:
        read_only = re.findall(r"const\s+\w+\s*\*\s*__restrict__\s+(\w+)", args)
        assert set(read_only) <= CALLERS, (kernel, read_only)
