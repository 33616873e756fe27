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


def _kernels(code):
    """(name, body) of every __global__ function."""
    for m in re.finditer(r"__global__", code):
        bounds = re.compile(r"__launch_bounds__\([^)]*\)").search(code, m.end(), m.end() + 80)
        head = re.compile(r"(\w+)\s*\(").search(code, bounds.end() if bounds else m.end())
        at = code.index("{", head.end())
        depth, i = 0, at
        while True:
            depth += {"{": 1, "}": -1}.get(code[i], 0)
            if depth == 0:
                break
            i += 1
        yield head.group(1), code[at + 1:i]


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_kernels_wait_for_their_asynchronous_copies_on_every_way_out(path):
    """A block's shared memory is another block's once it has left: where a kernel issues asynchronous copies, the wait for them stands at
    the outermost level behind the last of them, and nothing returns in between."""
    for name, body in _kernels(_code(path)):
        if "cp_async_16(" not in body:
            continue
        depth, waits = 0, []
        for m in re.finditer(r"[{}]|cp_async_wait_all\(\)", body):
            depth += {"{": 1, "}": -1}.get(m.group(), 0)
            if depth == 0 and m.group().startswith("cp_async"):
                waits.append(m.start())
        assert waits and waits[-1] > body.rindex("cp_async_16("), name
        assert not re.search(r"\breturn;", body[body.index("cp_async_16("):waits[-1]]), name


def test_the_rule_finds_the_kernels():
    found = {name for p in SOURCES for name, _ in _kernels(_code(p))}
    assert {"combine_splits_kernel", "token_logprob_kernel", "prune_fused_kernel", "column_sum_kernel"} <= found
