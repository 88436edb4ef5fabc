"""The deterministic engine's counters: (edge, vector) pairs and bytes of the pull count what it runs over -- every in-list
at depth 0, those of nodes with out-edges below -- before and after an update batch."""
import numpy as np
import pytest

from gpu_util import dedup
from paper_1709_06955_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_06955_gb300 import build
    build.build()


def dense_nodes(G, Q, l_max=64):
    """Columns pulled per depth: walk-tree nodes with a subtree of height >= 3, and super-roots (depth 0) of height >= 2."""
    nodes, lens = G.sample_walks(Q)
    height = {(): int(lens.max())}
    for w, length in zip(nodes.tolist(), lens.tolist()):
        for i in range(1, length + 1):
            key = tuple(w[:i])
            height[key] = max(height.get(key, 0), length - i)
    S = np.zeros(l_max + 2, np.int64)
    for key, h in height.items():
        S[len(key)] += h >= 3 or (not key and h >= 2)
    return S


def expected(n, s, d, S):
    out_deg, in_deg = np.bincount(s, minlength=n), np.bincount(d, minlength=n)

    def pieces(deg):
        return int(np.maximum(1, (deg + 127) // 128).sum())

    act = out_deg > 0
    gathers = nbytes = 0
    for depth, cols in enumerate(S.tolist()):
        if cols == 0:
            continue
        rows = in_deg if depth == 0 else in_deg[act]
        edges = int(rows.sum())
        gathers += edges * cols
        nbytes += 4 * edges + 16 * pieces(rows) + 4 * rows.size + 4 * cols * (int(act.sum()) + rows.size)
    return gathers, nbytes


def test_counters_follow_the_rows_pulled():
    from paper_1709_06955_gb300 import probesim
    n, s, d = synth.rmat(12, 6 << 12, seed=4)
    s, d = dedup(n, s, d)
    u = int(synth.queries(n, d, 1, seed=5)[0])
    Q = probesim.make_queries([u], eps=0.2, query_ids=[3])
    G = probesim.Graph(n, s, d)

    def check():
        G.single_source(Q)
        st = G.stats()
        gathers, nbytes = expected(n, s, d, dense_nodes(G, Q))
        assert st["edge_gathers"] == gathers
        assert st["probe_bytes"] == nbytes

    check()
    # a batch that takes edges away but leaves every node's out-list non-empty, so that the rows pulled stay the same nodes
    first = np.concatenate([[True], s[1:] != s[:-1]])
    cut = np.flatnonzero(~first)[::9]
    G.delete_edges(s[cut], d[cut])
    s, d = np.delete(s, cut), np.delete(d, cut)
    check()
    G.close()
