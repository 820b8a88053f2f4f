"""Memory ordering that no run shows reliably, read from the CUDA sources: a warp
refills a shared-memory slot, which all its lanes have read, by a bulk copy that
lane 0 issues.  The lanes' reads are ordered before the copy by __syncwarp()
alone; a vote (__all_sync) agrees on a value and orders no memory."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_14789_gb300", "csrc")


def _code(name):
    src = open(os.path.join(CSRC, name)).read()
    return re.sub(r"\s+", " ", re.sub(r"//[^\n]*|/\*.*?\*/", " ", src, flags=re.S))


@pytest.mark.parametrize("name,refills", [("kernels_warp.cu", 2), ("kernels_rbf_tiles.cu", 1)])
def test_every_refill_of_a_read_slot_follows_a_syncwarp(name, refills):
    code = _code(name)
    at = [m.start() for m in re.finditer(re.escape("if (lane == 0 && !last)"), code)]
    assert len(at) == refills
    for a in at:
        assert code[:a].rstrip().endswith("__syncwarp();"), code[max(0, a - 200):a + 60]
