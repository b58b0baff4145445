"""Kernels whose CTAs store into one another's shared memory, read as source:
no CTA leaves before every CTA of its cluster is past its last store, also when
a wait ran out.  So each of them ends with a cluster barrier that all its
threads reach, and none returns early once such stores may be under way."""
import glob
import os
import re

import pytest

from paper_2606_00946_gb300 import build as B

REMOTE = re.compile(r"seq_remote_store|st_async_|st_cluster_u32|ClusterRow|SentTotals|map_cluster|pair_stop")
CLOSING = re.compile(r"^  (?:if \(CL > 1\) )?cluster_sync\(\);", re.M)


def kernels():
    for path in sorted(glob.glob(os.path.join(B.CSRC, "*.cu"))):
        text = re.sub(r"//[^\n]*", "", open(path).read())
        for m in re.finditer(r"^__global__[^;{]*?\b(k_\w+)\s*\(.*?^}", text, re.M | re.S):
            yield m.group(1), m.group(0)


BODIES = {name: body for name, body in kernels() if REMOTE.search(body)}


def test_the_kernels_with_remote_stores_are_found():
    assert {"k_route_seq", "k_tr_chain", "k_score_pair"} <= set(BODIES)


@pytest.mark.parametrize("name", sorted(BODIES))
def test_ends_with_a_cluster_barrier(name):
    body = BODIES[name]
    last = max(m.end() for m in REMOTE.finditer(body))
    assert CLOSING.search(body, last), "no cluster barrier of all threads after the last remote store"
    first = CLOSING.search(body)
    assert not re.search(r"\breturn;", body[first.end():]), "a thread may leave early"
