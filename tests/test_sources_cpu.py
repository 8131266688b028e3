"""Rules of the CUDA programming model that no run can be relied on to show broken, checked on the sources."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2405_03133_b200", "csrc")


def kernels(name):
    """The __global__ functions of a file, comments removed: each from its qualifier to the next one's."""
    with open(os.path.join(CSRC, name)) as f:
        text = re.sub(r"//[^\n]*", "", f.read())
    return re.split(r"(?=__global__)", text)[1:]


@pytest.mark.parametrize("name", sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh"))))
def test_distributed_shared_memory_is_touched_after_a_cluster_barrier(name):
    """Another block's shared memory may be accessed only once that block is known to have started."""
    for body in kernels(name):
        if "map_shared_rank" in body:
            before = body[:body.index("map_shared_rank")]
            assert re.search(r"\.sync\(\)|barrier_wait\(", before), body[:200]


@pytest.mark.parametrize("name", sorted(n for n in os.listdir(CSRC) if n.endswith((".cu", ".cuh"))))
def test_no_mask_is_taken_from_whoever_happens_to_be_there(name):
    """__activemask() says which lanes are converged, not which will take part: no argument for a warp-wide exchange."""
    assert not any("__activemask" in body for body in kernels(name))
