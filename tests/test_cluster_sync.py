"""Distributed shared memory is touched only after a cluster barrier.

CUDA asks that every block of a cluster has started before another block accesses its shared
memory; being scheduled together does not say so.  No GPU: a missing barrier cannot be relied on to
show itself there, so the sources are read: between the start of a kernel and its first
map_shared_rank (or mapa) stands a cluster barrier's wait, and another one between its last and the
kernel's end.
"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2501_05587_gb300", "csrc")
BARRIER = re.compile(r"\.sync\(\)|\.barrier_wait\(|barrier\.cluster\.wait")
REMOTE = re.compile(r"\bmap_shared_rank\(|\bmapa\.")


def _kernels(text):
    """(name, body) of every __global__ function; // comments removed."""
    text = re.sub(r"//[^\n]*", "", text)
    for m in re.finditer(r"__global__", text):
        brace = text.index("{", m.end())
        depth, end = 0, brace
        while True:
            depth += {"{": 1, "}": -1}.get(text[end], 0)
            end += 1
            if depth == 0:
                break
        yield re.findall(r"(\w+)\s*\(", text[m.end():brace])[-1], text[brace:end]


@pytest.mark.parametrize("path", sorted(glob.glob(os.path.join(CSRC, "*.cu*"))), ids=os.path.basename)
def test_a_cluster_barrier_stands_before_and_after_remote_shared_memory(path):
    for name, body in _kernels(open(path).read()):
        uses = [m.start() for m in REMOTE.finditer(body)]
        if not uses:
            continue
        waits = [m.start() for m in BARRIER.finditer(body)]
        assert waits and min(waits) < uses[0], f"{name}: no cluster barrier before its first remote access"
        assert max(waits) > uses[-1], f"{name}: no cluster barrier after its last remote access"
