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
