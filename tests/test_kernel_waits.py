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


def test_no_thread_leaves_a_loop_by_its_own_wait():
    """The outcome of a bounded wait differs between threads when it runs out just as the copy lands, so
    it is agreed on (by the warp, the feeding warps or the block) before it decides about an exit: whoever
    stays would wait for those who left at the next barrier or shuffle, which has no limit."""
    for name, body in [(n, b) for _, n, b in _kernels() if "mbar_wait_bounded" in b]:
        for m in re.finditer(r"mbar_wait_bounded", body):
            start = max(body.rfind(c, 0, m.start()) for c in ";{}") + 1
            stmt = body[start:body.index(";", m.end()) + 1]
            tail = body[body.index(";", m.end()):]
            agreed = re.search(r"__syncthreads_and\s*\(\s*mbar_wait_bounded", stmt)
            kept = re.search(r"[^=!<>]=[^=]", stmt.split("mbar_wait_bounded")[0])
            alone = not re.search(r"\b(return|break)\b", stmt) and (not kept or re.search(r"feeders_agree<\w+>\(ok\)", tail))
            assert agreed or alone, (name, stmt.strip())


def test_named_barriers_carry_the_outcome():
    """A barrier among some of a block's warps is one that also says whether all of them go on."""
    for f in sorted(os.listdir(CSRC)):
        if f.endswith((".cu", ".cuh")):
            assert not re.search(r"bar(rier)?\.(cta\.)?sync", _source(f)), f


def test_an_exit_waits_for_its_copies():
    """Every warp that issues asynchronous copies gives those under way a bounded chance to land before it
    gives up: a copy that lands later writes into shared memory that belongs to another block by then."""
    issues = re.compile(r"bulk_load\s*\(|tma_load_2d\s*\(|tma_issue<\w+>\s*\(|pair_tile_issue<\w+>\s*\(|fetch_probe\s*\(")
    for name, body in [(n, b) for _, n, b in _kernels() if issues.search(b) and "mbar_wait" in b]:
        for m in re.finditer(r"if \(!(mbar_wait_warp|feeders_agree)[^{;]*([{;])", body):
            if m.group(2) == "{":
                block = body[m.end():body.index("}", m.end())]
                assert re.search(r"mbar_wait_bounded|drain", block), (name, m.group(0))
            else:                                      # a warp that issues none: its block's feeders drain
                assert re.search(r"if \(!feeders_agree<\w+>\(ok\)\) {\s*drain_fetch", body), (name, m.group(0))
        if "__syncthreads_and" in body:
            after = body[body.index("__syncthreads_and"):]
            assert re.search(r"if \((threadIdx\.x == 0|!ok)[^;]*\)?\s*mbar_wait_bounded", after), name
