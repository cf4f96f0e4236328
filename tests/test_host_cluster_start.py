"""A block's shared memory may be accessed by the other blocks of its cluster only once it has started, which a cluster
barrier tells. In every kernel that reaches into other blocks, such a barrier comes before the first access (a helper that
sums over the cluster has one before it reads). Checked on the source: started too early, a block would be written before
its time only now and then."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1402_0266_gb300", "csrc")
# arrival alone is no barrier; mapping a pointer (p = cl.map_shared_rank(...)) is no access
BARRIER = re.compile(r"\bcl\.sync\(\)|\bcl\.barrier_wait\(\)|\bcluster_sum[24]\(cl")
ACCESS = re.compile(r"(?<![=?] )\bcl\.map_shared_rank\(")


def _functions(name):
    """Bodies of the file's functions, comments taken out: a definition ends with a brace in the first column."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, name)).read())
    return [b for b in re.split(r"\n}", text) if "map_shared_rank" in b]


def _sources():
    return [f for f in sorted(os.listdir(CSRC)) if "map_shared_rank" in open(os.path.join(CSRC, f)).read()]


@pytest.mark.parametrize("name", _sources())
def test_a_cluster_barrier_comes_before_the_first_remote_access(name):
    for body in _functions(name):
        access = ACCESS.search(body)
        if not access:
            continue
        barrier = BARRIER.search(body)
        assert barrier and barrier.start() < access.start(), body[max(0, access.start() - 200):access.end() + 60]
