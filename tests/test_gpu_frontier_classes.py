"""Every class of the frontier engine's tables at its bounds, against the oracle.  The frontiers of every probe are formed
here as sets, so it is known which class each next frontier falls in, and that the intended one runs; the bounds come from
the source."""
import os
import re

import numpy as np
import pytest

from gpu_util import TOL, dedup, oracle_graph
from test_gpu_frontier_global import two_hubs

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_06955_gb300", "csrc")
with open(os.path.join(CSRC, "internal.cuh")) as _f:
    _TEXT = _f.read()
WARP, BLOCK, MID, PART, SLAB, SLAB_PARTS, PARTS = (
    int(re.search(r"\b%s = (\d+)" % k, _TEXT).group(1))
    for k in ("kWarpD", "kBlockD", "kMidD", "kPartD", "kSlabN", "kSlabParts", "kMaxParts"))


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_06955_gb300 import build
    from oracle import build as obuild
    build.build()
    obuild.build()


def class_of(items, entries, last, n):
    """The class of a probe's level, as the planner's comment states it."""
    D = min(items, n)
    if last:
        return "last"
    if entries == 1:
        return "single"
    if D <= WARP:
        return "warp"
    if D <= BLOCK:
        return "block"
    if 4 * D >= n and n <= SLAB * SLAB_PARTS:
        return "slab"
    if D <= MID:
        return "mid"
    if D <= PART * PARTS:
        return "wide%d" % -(-D // PART)
    return "dense" if 4 * D >= n else "hash"


def levels_of(n, s, d, walks, lens):
    """(class, items) of every level of every probe, and the sum of the items."""
    start, out = np.searchsorted(s, np.arange(n + 1)), d[np.argsort(s, kind="stable")]
    prefixes = {tuple(w[:q]) for w, l in zip(walks.tolist(), lens.tolist()) for q in range(2, l + 1)}
    seen, total = {}, 0
    for pre in prefixes:
        q, frontier = len(pre), np.array([pre[-1]])
        for j in range(q - 1):
            frontier = frontier[start[frontier + 1] > start[frontier]]
            if frontier.size == 0:
                break
            targets = np.concatenate([out[start[x]:start[x + 1]] for x in frontier]) if frontier.size < 4 else \
                out[np.repeat(start[frontier], start[frontier + 1] - start[frontier]) + _within(start, frontier)]
            total += targets.size
            c = class_of(targets.size, frontier.size, j == q - 2, n)
            seen.setdefault(c, set()).add(min(targets.size, n))
            frontier = np.unique(targets[targets != pre[q - j - 2]])
    return seen, total


def _within(start, nodes):
    deg = start[nodes + 1] - start[nodes]
    return np.arange(deg.sum()) - np.repeat(np.cumsum(deg) - deg, deg)


def check(n, s, d, u, want, walk_end=32):
    """All-deterministic switch mode (c0 huge); `want`: classes that must run, with the bound on the next frontier."""
    from paper_1709_06955_gb300 import probesim
    s, d = dedup(n, s, d)
    G = probesim.Graph(n, s, d, probe_mode=probesim.PROBE_SWITCH, c0=1e30)
    Q = probesim.make_queries([u], eps=0.2, query_ids=[81], walk_begin=0, walk_end=walk_end)
    got = G.single_source(Q)[0]
    pushes = G.stats()["edge_gathers"]
    walks, lens = G.sample_walks(Q)
    G.close()
    seen, total = levels_of(n, s, d, walks, lens)
    for c, D in want:
        assert D in seen.get(c, ()), (c, D, seen)
    assert pushes == total
    ref, _ = oracle_graph(n, s, d).single_source(u, eps=0.2, seed=3, qid=81, walk_begin=0, walk_end=walk_end)
    assert np.max(np.abs(got - ref)) <= TOL


def bounds():
    big = 4 * (PART * PARTS + 2) + 17  # more than four times any bound: no slabs
    rows = []
    for D, c in [(WARP, "warp"), (WARP + 1, "block"), (BLOCK, "block"), (BLOCK + 1, "mid"), (MID, "mid"),
                 (MID + 1, "wide1"), (PART, "wide1"), (PART + 1, "wide2"), (2 * PART, "wide2"), (2 * PART + 1, "wide3"),
                 (PART * PARTS, "wide%d" % PARTS), (PART * PARTS + 1, "hash")]:
        rows.append((big, D, c))
    n = SLAB * SLAB_PARTS  # the largest graph with slabs, and one node more
    rows += [(n, n // 4, "slab"), (n, n // 4 - 1, "wide%d" % -(-(n // 4 - 1) // PART)),
             (n + 1, n // 4 + 1, "wide%d" % -(-(n // 4 + 1) // PART)), (n + 1, PART * PARTS + 1, "dense"),
             (4 * (PART * PARTS + 1), PART * PARTS + 1, "dense"), (4 * (PART * PARTS + 1) + 1, PART * PARTS + 1, "hash"),
             (SLAB, BLOCK + 1, "mid"), (SLAB, SLAB // 4, "slab"), (SLAB + 1, SLAB // 2, "slab")]
    return rows


@pytest.mark.parametrize("n,D,cls", bounds())
def test_class_at_its_bound(n, D, cls):
    fa = D // 2 + D // 6
    s, d, (u,) = two_hubs(n, [(fa, D - fa)])
    check(n, s, d, u, [(cls, D)])


def _mix32(h):
    h = h.astype(np.uint64)
    m = np.uint64(0xFFFFFFFF)
    h ^= h >> np.uint64(16)
    h = (h * np.uint64(0x85EBCA6B)) & m
    h ^= h >> np.uint64(13)
    h = (h * np.uint64(0xC2B2AE35)) & m
    return h ^ (h >> np.uint64(16))


@pytest.mark.parametrize("n,k,bits", [(80000, 17000, 1), (260000, 20000, 3)])
def test_a_part_with_more_nodes_than_its_table_has_slots(n, k, bits):
    """k distinct targets, more than the 16,384 slots of a table, whose hashes share their top bits: all in the first of two
    parts, which is split in halves until it fits (twice and more with three common bits)."""
    a, b, c, u = 0, 1, 2, 9
    ids = np.arange(10, n)
    hit = ids[(_mix32(ids) >> np.uint64(32 - bits)) == 0][:k]
    assert hit.size == k > 16384 and PART < k <= 2 * PART and 4 * k < n
    # internal ids are the caller's here: nodes 0..3 have the largest out-degrees in order, every other node one out-edge
    fa = k // 2 + 100
    rest = np.setdiff1d(np.arange(n), [a, b, c, 3])
    src = [np.full(fa - 1, a), np.full(k - fa - 1, b), [a, b, c, c, c, 3, 3], rest]
    dst = [hit[:fa - 1], hit[fa - 1:k - 2], [u, u, a, b, 3, c, hit[0]], np.where(rest == 5, 6, 5)]
    check(n, np.concatenate(src), np.concatenate(dst), u, [("wide2", k)])
