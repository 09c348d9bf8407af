"""Rules that the kernels' sources keep because breaking one hangs or faults a GPU only now and then: read here, not run."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_26558_b200", "csrc")
SOURCES = sorted(f for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh")))


def _functions(name):
    """Top-level blocks of a source without its comments: each ends with a closing brace in the first column."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    return re.split(r"\n}[^\n]*\n", text)


@pytest.mark.parametrize("name", SOURCES)
def test_distributed_shared_memory_is_touched_behind_a_cluster_barrier(name):
    """A CTA's shared memory may be read or written by others of its cluster only once it is known to run."""
    for body in _functions(name):
        first = body.find("map_shared_rank")
        if first >= 0:
            assert re.search(r"cluster\.(sync|barrier_wait)\(\)", body[:first]), body[:200]


@pytest.mark.parametrize("name", SOURCES)
def test_who_gives_up_still_meets_the_cluster(name):
    """A thread that gives up a bounded wait and goes straight to the cluster's barrier leaves the others of its CTA at
    __syncthreads, and the cluster waits for them for good: its warp decides as one and stays on the way that all take."""
    for body in _functions(name):
        if "mbar_wait_bounded(" in body and re.search(r"cluster\.(sync|barrier_arrive|barrier_wait)\(\)", body):
            gives_up = re.search(r"\n( +)if \(!mbar_wait_bounded\([^;{]*\{(.*?)\n\1\}\n +lost = __any_sync\(0xffffffffu, lost\);", body, re.S)
            assert gives_up and re.findall(r"\n *(.*)return", gives_up[2]) == ["if (out != 2) "], body[:200]


@pytest.mark.parametrize("name", SOURCES)
def test_copies_in_flight_land_before_their_block_ends(name):
    """A kernel that gives up a wait for a copy waits (again with a limit, whatever the outcome) for the copies it has started: they
    would land in the shared memory of the block after it."""
    for body in _functions(name):
        if "__global__" in body and re.search(r"\b(tma_load_\dd|bulk_g2s)\(", body):
            assert re.search(r"\n +mbar_wait_bounded\(", body), body[:200]
