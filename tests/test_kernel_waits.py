"""Waits of the kernels, read from their source (no GPU): what a run that goes well never shows.

A missing wait or an exit that leaves a copy in flight cannot be shown by running it: it goes well
nearly always, and where it does not, the GPU is what suffers."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2311_14780_gb300", "csrc")


def _source(name):
    text = open(os.path.join(CSRC, name)).read()
    return re.sub(r"//[^\n]*", "", text)


def _bodies(text):
    """(name, body) of every kernel in a source text."""
    out = []
    for m in re.finditer(r"__global__[^;{]*?\b(k_\w+)\s*\(", text):
        i = text.find("{", m.end())
        semi = text.find(";", m.end())
        if i < 0 or 0 <= semi < i:
            continue                                                       # a declaration
        depth, j = 1, i + 1
        while depth:
            depth += {"{": 1, "}": -1}.get(text[j], 0)
            j += 1
        out.append((m.group(1), text[i:j]))
    return out


def _kernels():
    return [(f, n, b) for f in sorted(os.listdir(CSRC)) if f.endswith((".cu", ".cuh")) for n, b in _bodies(_source(f))]


def test_another_blocks_shared_memory_only_after_a_cluster_barrier():
    """Distributed shared memory may be accessed once every block of the cluster has started."""
    users = [(n, b) for _, n, b in _kernels() if "map_shared_rank" in b]
    assert users
    for name, body in users:
        before = body[:body.index("map_shared_rank")]
        assert re.search(r"\.(barrier_wait|sync)\s*\(", before), name
