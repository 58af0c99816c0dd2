"""Distributed shared memory may be touched only while the CTA it belongs to is running: every kernel
that stores into or loads from another CTA of its cluster completes a cluster barrier first.  Checked on
the sources, since a run on the GPU shows only its usual timing."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1508_07621_gb300", "csrc")
REMOTE = re.compile(r"\b(?:st|ld)\.shared::cluster\.|\bst_cluster_\w+\(|\bld_cluster\(|\boz_fold\(")
BARRIER = re.compile(r"barrier\.cluster\.wait|\bcluster_sync_all\(|\boz_cluster_sync\(|\bcluster_wait\(")


def _kernels():
    """(name, body) of every __global__ function of the sources, comments removed."""
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))):
        with open(path) as f:
            text = re.sub(r"//[^\n]*", "", f.read())
        for m in re.finditer(r"__global__", text):
            head = text.index("{", m.end())
            depth, end = 0, head
            while True:
                depth += {"{": 1, "}": -1}.get(text[end], 0)
                end += 1
                if depth == 0:
                    break
            name = re.search(r"\bk_\w+", text[m.end():head])
            if name:
                yield name.group(0), text[head:end]


CLUSTERED = {name: body for name, body in _kernels() if REMOTE.search(body)}


def test_clustered_kernels_are_found():
    assert {"k_dense_resident", "k_dense_resident_dfl", "k_oz_term", "k_oz_real_term"} <= set(CLUSTERED)


@pytest.mark.parametrize("name", sorted(CLUSTERED))
def test_cluster_barrier_before_remote_access(name):
    body = CLUSTERED[name]
    barrier = BARRIER.search(body)
    assert barrier and barrier.start() < REMOTE.search(body).start()
