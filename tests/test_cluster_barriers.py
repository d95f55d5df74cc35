"""Kernels of a thread-block cluster may touch another block's shared memory only once every block of the cluster is known to have
started (and only until one of them may have left).  The first half is read off the sources: in every kernel that maps shared memory of
another block, a barrier of the cluster comes before the first use of such a mapping."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_20787_b200", "csrc")


def _kernels():
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        starts = [m.start() for m in re.finditer(r"__global__", text)] + [len(text)]
        for a, b in zip(starts, starts[1:]):
            if "map_shared_rank" in text[a:b]:
                yield os.path.basename(path), re.search(r"(\w+)\s*\(\s*(?:const|unsigned)", text[a:b]).group(1), text[a:b]


KERNELS = {"%s:%s" % (f, name): body for f, name, body in _kernels()}


@pytest.mark.parametrize("kernel", sorted(KERNELS))
def test_cluster_has_started_before_remote_shared_memory(kernel):
    body = KERNELS[kernel]
    barrier = re.search(r"cluster\.(sync|barrier_wait)\s*\(", body)
    assert barrier and barrier.start() < body.index("map_shared_rank")
    if "barrier_wait" in body:
        assert body.index("barrier_arrive") < body.index("barrier_wait")
