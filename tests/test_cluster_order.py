"""Order of the cluster barriers in the kernel sources.  A CTA may write into another CTA's shared memory only when that CTA
is known to run: every kernel that does must have passed a cluster barrier (an arrival and a wait by all its threads) before
its first remote store.  Nothing on the device reports a store that came too early, so the order is read off the source."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_07355_b200", "csrc")


def kernels():
    """(name, body without comments) of every kernel"""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for part in text.split("__global__")[1:]:
            name = re.search(r"\b(k_\w+)\s*\(", part).group(1)
            start = part.index("{", part.index(name))
            depth, end = 0, start
            for end in range(start, len(part)):
                depth += {"{": 1, "}": -1}.get(part[end], 0)
                if depth == 0:
                    break
            yield name, part[start:end]


CLUSTERED = [(n, b) for n, b in kernels() if "st_cluster_" in b]


def test_the_kernels_that_store_remotely_are_found():
    assert {"k_match_tc", "k_frame_stats_cluster", "k_stats_cluster"} <= {n for n, _ in CLUSTERED}


@pytest.mark.parametrize("name,body", CLUSTERED, ids=[n for n, _ in CLUSTERED])
def test_a_cluster_barrier_precedes_the_first_remote_store(name, body):
    first = body.index("st_cluster_")
    assert 0 <= body.find("cluster_arrive()") < body.find("cluster_wait()") < first
    last = body.rindex("st_cluster_")                        # and one follows the last, before anybody reads
    assert last < body.rindex("cluster_arrive()") < body.rindex("cluster_wait()")
