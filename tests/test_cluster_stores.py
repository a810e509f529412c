"""Remote shared memory: a CTA of a cluster may be written only once it is known to run.

The order cannot be made to fail on demand, so it is read from the sources: every kernel
that maps another CTA's shared memory has arrived at a cluster barrier and waited on it
before, and passes a second barrier after.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2312_10044_gb300", "csrc")


def _kernels():
    """(file:kernel, body) of every kernel that maps remote shared memory."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for part in re.split(r"(?=__global__)", text)[1:]:
            name = re.search(r"\b(k_\w+)\s*\(", part).group(1)
            start = part.index("{", part.index(")", part.index(name)))
            depth, end = 0, start
            for end in range(start, len(part)):
                depth += {"{": 1, "}": -1}.get(part[end], 0)
                if depth == 0:
                    break
            body = part[start:end]
            if "map_shared_rank" in body:
                yield f"{os.path.basename(path)}:{name}", body


KERNELS = dict(_kernels())


def test_kernels_are_found():
    assert {"kernels.cu:k_reduce_reaction", "mrhs_tc.cu:k_colmax_u"} <= set(KERNELS)


@pytest.mark.parametrize("name", sorted(KERNELS))
def test_remote_stores_follow_a_cluster_wait(name):
    body = KERNELS[name]
    first, last = body.index("map_shared_rank"), body.rindex("map_shared_rank")
    waits = [m.start() for m in re.finditer(r"cluster_wait\(\)|cluster_sync\(\)|\.sync\(\)", body)]
    arrives = [m.start() for m in re.finditer(r"cluster_arrive\(\)|cluster_sync\(\)|\.sync\(\)", body)]
    assert waits and arrives and arrives[0] <= waits[0] < first, "stores before the other CTA is known to run"
    assert waits[-1] > last, "the stores are not made visible"
