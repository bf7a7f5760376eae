"""Thread-block clusters, checked in the source (the fault is a race that need not show on a GPU): a
block's shared memory may be accessed by another block of its cluster only once that block has
started, which a cluster barrier completed before the access establishes."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1804_01184_gb300", "csrc")


def kernels():
    """(file, name, body) of every __global__ function with a body, comments removed."""
    for f in sorted(os.listdir(CSRC)):
        src = open(os.path.join(CSRC, f)).read()
        src = re.sub(r"//[^\n]*|/\*.*?\*/", "", src, flags=re.S)
        for m in re.finditer(r"__global__", src):
            head = re.compile(r"(\w+)\s*\((?:[^(){};]|\([^()]*\))*\)\s*\{").search(src, m.end())
            if not head:
                continue
            depth, end = 1, head.end()
            while depth and end < len(src):
                depth += {"{": 1, "}": -1}.get(src[end], 0)
                end += 1
            yield f, head.group(1), src[head.end():end]


REMOTE = re.compile(r"map_shared_rank\s*\(|\bmapa\b|shared::cluster")
BARRIER = re.compile(r"\.barrier_wait\s*\(|barrier\.cluster\.wait|\bcl\.sync\s*\(")


def remote_kernels():
    return [(f, n, b) for f, n, b in kernels() if "map_shared_rank" in b]


def test_kernels_are_found():
    names = [n for _, n, _ in kernels()]
    assert "k_misfit" in names and "k_model" in names
    assert [n for _, n, _ in remote_kernels()] == ["k_misfit"]


@pytest.mark.parametrize("case", remote_kernels(), ids=lambda c: c[1])
def test_a_cluster_barrier_completes_before_the_first_remote_access(case):
    _, _, body = case
    first = REMOTE.search(body).start()
    assert BARRIER.search(body[:first]), "remote shared memory is accessed before any cluster barrier"
    assert BARRIER.search(body[first:]), "the target block may exit before its memory has been accessed"
