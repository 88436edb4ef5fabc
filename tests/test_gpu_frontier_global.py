"""The frontier engine's tables in device memory, which calls of one graph keep: a call that needs more slots than the one
before, against the call alone on a fresh graph (bit for bit: its sums are exact) and against the oracle."""
import numpy as np
import pytest

from gpu_util import TOL, dedup, oracle_graph

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


def two_hubs(n, fans):
    """Per pair (fa, fb) of `fans`: u <- a, b <- c <-> d with |O(a)| = fa, |O(b)| = fb and overlapping targets, each of
    which has one out-edge.  The probe of (u, a, c, d, c) has the frontier {a, b} at level 1, so its next frontier's bound
    is fa + fb.  Returns the edges and the nodes u."""
    src, dst, roots, at = [], [], [], 5 * len(fans)
    for k, (fa, fb) in enumerate(fans):
        a, b, c, d, u = range(5 * k, 5 * k + 5)
        roots.append(u)
        ta, tb = at + np.arange(fa - 1), at + (fa - 1) // 2 + np.arange(fb - 1)
        ring = np.arange(at, max(ta[-1], tb[-1]) + 1)
        at = int(ring[-1]) + 1
        src += [np.full(fa - 1, a), np.full(fb - 1, b), ring, [a, b, c, c, c, d]]
        dst += [ta, tb, np.roll(ring, 1), [u, u, a, b, d, c]]
    assert at <= n
    return dedup(n, np.concatenate(src), np.concatenate(dst)) + (roots,)


def test_table_grows_between_calls():
    """80,000 and 200,000 entries of a million nodes: 2^18 and 2^19 slots a probe, above the tables in shared memory."""
    from paper_1709_06955_gb300 import probesim
    n = 1_000_000
    s, d, roots = two_hubs(n, [(50000, 30000), (110000, 90000)])

    def graph():
        return probesim.Graph(n, s, d, probe_mode=probesim.PROBE_SWITCH, c0=1e30)

    def query(G, u):
        return G.single_source(probesim.make_queries([u], eps=0.2, query_ids=[81], walk_begin=0, walk_end=40))[0]

    G = graph()
    got, slots = [], []
    for u in roots:
        got.append(query(G, u))
        slots.append(G.stats()["max_table_slots"])
    again = query(G, roots[0])
    G.close()
    assert slots[0] >= 1 << 18 and slots[1] >= 1 << 19
    assert np.array_equal(again, got[0])
    O = oracle_graph(n, s, d)
    for u, x in zip(roots, got):
        F = graph()
        assert np.array_equal(query(F, u), x)
        F.close()
        ref, _ = O.single_source(u, eps=0.2, seed=3, qid=81, walk_begin=0, walk_end=40)
        assert np.max(np.abs(x - ref)) <= TOL
