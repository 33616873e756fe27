"""Rules of the kernels' sources that no run can be relied on to show."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_24840_b200", "csrc")
SOURCES = sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")))
ALIGNED_BARRIER = re.compile(r'asm volatile\(\s*"(bar\.(sync|arrive)\b|barrier\.cluster\.(arrive|wait)\S*\.aligned|'
                             r'tcgen05\.(alloc|dealloc|relinquish_alloc_permit)\b)')


def _code(path):
    return re.sub(r"//[^\n]*", "", open(path).read())


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_aligned_barriers_follow_a_warp_barrier(path):
    """The aligned barriers, and the allocation of tensor memory, are undefined in a warp that is not converged: each is issued directly
    behind a __syncwarp()."""
    code = _code(path)
    for m in ALIGNED_BARRIER.finditer(code):
        assert code[:m.start()].rstrip().endswith("__syncwarp();"), "%s: %s" % (os.path.basename(path), code[m.start():m.start() + 80])


def test_the_rule_finds_the_barriers():
    assert sum(len(ALIGNED_BARRIER.findall(_code(p))) for p in SOURCES) >= 10
