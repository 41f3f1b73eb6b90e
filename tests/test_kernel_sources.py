"""Orderings that a run on the GPU shows only by chance, read from the kernels'
sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_07993_gb300", "csrc")


def kernels():
    """(file, body) of every __global__ function."""
    for f in sorted(os.listdir(CSRC)):
        if not f.endswith((".cu", ".cuh")):
            continue
        text = open(os.path.join(CSRC, f)).read()
        for m in re.finditer(r"__global__", text):
            a = text.index("{", m.end())
            depth, b = 0, a
            while True:
                depth += {"{": 1, "}": -1}.get(text[b], 0)
                b += 1
                if depth == 0:
                    break
            yield f, text[a:b]


def test_remote_shared_memory_between_cluster_barriers():
    """A CTA's shared memory may be written from another CTA of its cluster
    only once it is known to run, and read there only after the writers: a
    cluster barrier's arrive and wait before the first remote store, and
    another pair after the last."""
    seen = 0
    for f, body in kernels():
        stores = [m.start() for m in re.finditer(r"st\.shared::cluster", body)]
        if not stores:
            continue
        seen += 1
        for word in (r"barrier\.cluster\.arrive", r"barrier\.cluster\.wait"):
            at = [m.start() for m in re.finditer(word, body)]
            assert any(a < stores[0] for a in at), f"{f}: no {word} before the first remote store"
            assert any(a > stores[-1] for a in at), f"{f}: no {word} after the last remote store"
    assert seen
