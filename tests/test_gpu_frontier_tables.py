"""The frontier engine's tables: next-frontier bounds on both sides of every class (warp, block, wide in parts, global,
dense), parts that hold more nodes than a table, and deferred ranges, against the oracle and against each other."""
import numpy as np
import pytest

from gpu_util import TOL, dedup, oracle_graph
from paper_1709_06955_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_06955_gb300 import build
    from oracle import build as obuild
    build.build()
    obuild.build()


def _check(n, s, d, u, walks, eps_p=0.0, budget=0):
    """All-deterministic switch mode (c0 huge), so every prefix runs through the tables."""
    from paper_1709_06955_gb300 import probesim
    s, d = dedup(n, s, d)
    G = probesim.Graph(n, s, d, probe_mode=probesim.PROBE_SWITCH, c0=1e30, eps_p=eps_p)
    Q = probesim.make_queries([u], eps=0.2, query_ids=[81], walk_begin=0, walk_end=walks)
    got = G.single_source(Q)[0]
    stats = G.stats()
    if budget:
        G.set_memory_budget(budget)
        assert np.array_equal(G.single_source(Q)[0], got)
        assert G.stats()["deferred"] > 0
    G.close()
    ref, _ = oracle_graph(n, s, d).single_source(u, eps=0.2, seed=3, qid=81, walk_begin=0, walk_end=walks)
    if eps_p:  # every pruned level takes at most eps_p from a walk's estimate
        assert np.all(got <= ref + TOL)
        return got, stats
    assert np.max(np.abs(got - ref)) <= TOL
    return got, stats


@pytest.mark.parametrize("fan", [3, 63, 64, 65, 511, 512, 513, 2047, 2048, 2049, 8191, 8193, 32767, 32769, 40000])
def test_classes_at_their_bounds(fan):
    """u <- a, b <- c <-> d: the walks reach c through a and b; the probes of the longer prefixes have two entries (a and
    b) whose out-lists overlap, so the next frontier's bound is 2 fan."""
    a, b, c, d, u = 0, 1, 2, 3, 4
    n = max(5 + 3 * fan // 2 + 10, 100)
    t = np.arange(5, 5 + fan)
    src = [[a, b, c, c, d, a, b], np.full(fan, a), np.full(fan, b)]
    dst = [[u, u, a, b, c, u, u], t, t + fan // 2]
    back = np.arange(5, 5 + 3 * fan // 2)
    src.append(back)  # the targets go on, so that their sums are pushed once more
    dst.append(np.where(back % 7 == 0, c, back - 1))
    src.append([c])
    dst.append([d])
    _check(n, np.concatenate(src), np.concatenate(dst), u, 48)


def _mix32(h):
    h = h.astype(np.uint64)
    m = np.uint64(0xFFFFFFFF)
    h ^= h >> np.uint64(16)
    h = (h * np.uint64(0x85EBCA6B)) & m
    h ^= h >> np.uint64(13)
    h = (h * np.uint64(0xC2B2AE35)) & m
    return h ^ (h >> np.uint64(16))


def test_a_part_larger_than_its_table_is_split():
    """Targets chosen so that their hashes share the top two bits: 9,000 nodes in one part of 8,192 slots."""
    k = 9000
    n = 80000
    ids = np.arange(10, n)
    hit = ids[(_mix32(ids) >> np.uint64(30)) == 1][:k]
    assert hit.size == k
    # ids are internal ids here: nodes 0..3 have the largest out-degrees in order, every other node has out-degree 1
    a, b, c, u = 0, 1, 2, 9
    src = [np.full(k, a), np.full(k - 500, b), np.full(40, c)]
    dst = [hit, hit[250:k - 250], np.arange(n - 40, n)]
    src += [[a, b, c, c]]
    dst += [[u, u, a, b]]
    rest = np.setdiff1d(np.arange(n), [a, b, c])
    src.append(rest)
    dst.append(np.where(rest == 5, 6, 5))
    src.append([3])
    dst.append([c])
    _check(n, np.concatenate(src), np.concatenate(dst), u, 32)


@pytest.mark.parametrize("scale,deg,eps_p", [(12, 24, 0.0), (13, 16, 3.1e-4), (17, 16, 0.0)])
def test_random_graphs_and_deferred_ranges(scale, deg, eps_p):
    n, s, d = synth.rmat(scale, deg << scale, seed=scale)
    n -= 37  # not a power of two
    keep = (s < n) & (d < n)
    s, d = s[keep], d[keep]
    u = int(synth.queries(n, d, 1, seed=5)[0])
    _check(n, s, d, u, 40, eps_p, budget=160 * n)


def test_scores_that_round_to_zero_stay_members():
    """Hubs of in-degree about 1,000 in a row divide a score below the fixed-point unit; its node stays a member and is
    pushed on, so the engine's count of pushes equals that of the frontier sets."""
    from paper_1709_06955_gb300 import probesim
    steps, width, fans = 9, 3, 900
    edges, nxt = [], 0

    def new(k):
        nonlocal nxt
        nxt += k
        return np.arange(nxt - k, nxt)

    chain = new(steps + 2)  # the walk: chain[0] <- chain[1] <- ...
    edges += [(chain[i + 1], chain[i]) for i in range(steps + 1)]
    prev = [chain[-1]]
    for _ in range(steps):  # layers of hubs, each fed by the previous layer and by dummies
        layer = new(width)
        for h in layer:
            edges += [(x, h) for x in prev] + [(x, h) for x in new(fans // width)]
        leaves = new(700)  # wide out-lists keep the frontier's bound above a quarter of the nodes
        edges += [(h, v) for h in layer for v in leaves]
        prev = list(layer)
    n = nxt
    s, d = dedup(n, *np.array(edges, np.int64).T)
    out = [[] for _ in range(n)]
    for a, b in zip(s, d):
        out[a].append(b)
    G = probesim.Graph(n, s, d, probe_mode=probesim.PROBE_SWITCH, c0=1e30)
    Q = probesim.make_queries([int(chain[0])], eps=0.2, query_ids=[9], walk_begin=0, walk_end=400)
    G.single_source(Q)
    pushes = G.stats()["edge_gathers"]
    nodes, lens = G.sample_walks(Q)
    G.close()
    prefixes = {tuple(w[:q]) for w, l in zip(nodes.tolist(), lens) for q in range(2, l + 1)}
    assert max(len(x) for x in prefixes) >= steps  # some walk is long enough to reach the small scores
    want = 0
    for pre in prefixes:
        frontier = {pre[-1]}
        for j in range(len(pre) - 1):
            want += sum(len(out[x]) for x in frontier)
            frontier = {v for x in frontier for v in out[x] if v != pre[len(pre) - j - 2]}
    assert pushes == want


@pytest.mark.parametrize("n", [7001, 24576, 24577, 98305, 245760, 245761])
def test_last_level_summed_in_shared_memory(n):
    """One query's last-level pushes are summed in slabs of 24,576 nodes in shared memory (on a graph of at most ten of
    them), several queries' straight in the estimates: the sums are exact, so the estimates are equal bit for bit."""
    from paper_1709_06955_gb300 import probesim
    rng = np.random.default_rng(n)
    m = 16 * n
    s = rng.permutation(n)[(n * rng.random(m) ** 3).astype(np.int64)]
    d = rng.permutation(n)[(n * rng.random(m) ** 2).astype(np.int64)]
    s, d = dedup(n, s, d)
    sp = probesim.split_error(0.1, c=0.6, shift=True)
    G = probesim.Graph(n, s, d, l_max=sp["l_max"], eps_p=sp["eps_p"], shift=sp["shift"])
    nodes = [int(x) for x in rng.choice(np.unique(d), 2, replace=False)]
    ids = np.array([5, 6])
    both = G.single_source(probesim.make_queries(nodes, eps=sp["eps"], query_ids=ids))
    for i in range(2):
        alone = G.single_source(probesim.make_queries(nodes[i:i + 1], eps=sp["eps"], query_ids=ids[i:i + 1]))
        assert np.array_equal(alone[0], both[i])
    G.close()
