"""Bounded waits of the tensor-memory kernels: where a warp's lanes work together after a wait (tensor-memory loads,
shuffles, __syncwarp), no lane can leave alone."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1503_01722_gb300", "csrc")
TOGETHER = re.compile(r"tmem_ld16\(|__shfl|__syncwarp\(")


def blocks(s, head):
    """The bodies of the braces that follow each match of head."""
    for m in re.finditer(head, s):
        i = s.index("{", m.end() - 1)
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(s[j], 0)
            j += 1
        yield m.group(0), s[i:j]


@pytest.mark.parametrize("name,loops", [("ocmc_unet_tc.cu", 3), ("ocmc_unet_wgrad_tc.cu", 2)])
def test_loops_that_a_warp_leaves_together(name, loops):
    with open(os.path.join(CSRC, name)) as f:
        s = re.sub(r"//[^\n]*", "", f.read())
    for head, body in blocks(s, r"for \([^{}]*?\*abort[^{}]*?\{"):
        assert not TOGETHER.search(body), (head, body)       # a lane's own look at the flag, work together inside
    seen = 0
    for head, body in blocks(s, r"(?:for \((?:int tile|long long i) = [^{}]*?|if \(mbar_wait\w*\(done[^{}]*?)\{"):
        if TOGETHER.search(body):
            seen += 1
            for wait in re.findall(r"mbar_wait\w*\([^;]*", head + body):
                if "empty" not in wait:                      # one lane's wait, its answer broadcast
                    assert wait.startswith("mbar_wait_warp("), wait
    assert seen >= loops
