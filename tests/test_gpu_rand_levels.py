"""The randomized PROBE's level lists: node records at the edges of their 8-bit ids, lists that a level outgrows, and
entries on both sides of the warp's one-entry path, against the oracle (exact integer member counts)."""
import numpy as np
import pytest

from gpu_util import dedup, oracle_graph
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


def _counts_equal(n, s, d, nodes, eps, budget=0):
    from paper_1709_06955_gb300 import probesim
    s, d = dedup(n, s, d)
    G = probesim.Graph(n, s, d, probe_mode=probesim.PROBE_RANDOMIZED)
    if budget:
        G.set_memory_budget(budget)
    O = oracle_graph(n, s, d)
    out = G.single_source(probesim.make_queries(nodes, eps=eps, query_ids=np.arange(len(nodes)) + 70))
    nr = G.num_walks(eps)
    for t, u in enumerate(nodes):
        ref, _ = O.single_source(int(u), eps=eps, seed=3, qid=70 + t, probe_mode=1)
        got = np.rint(out[t].astype(np.float64) * nr)
        want = np.rint(ref * nr)
        got[u] = want[u] = 0
        assert np.array_equal(got, want)
    G.close()


@pytest.mark.parametrize("n", [2, 255, 256, 257, 511, 513, 1023])
def test_record_ids_at_the_shift_boundaries(n):
    rng = np.random.default_rng(n)
    k = 1 if n == 2 else 9 * n
    s, d = rng.integers(0, n, k), rng.integers(0, n, k)
    s[0], d[0] = 0, 1
    _counts_equal(n, s, d, [1, n - 1], 0.3)


@pytest.mark.parametrize("fan", [31, 32, 33, 63, 64, 65, 2500])
@pytest.mark.parametrize("budget", [0, 1 << 20])
def test_members_that_outgrow_the_list(fan, budget):
    """Children of in-degree 1 are members three times out of four; a dense part elsewhere makes the graph's mean, which
    sizes the lists, small.  Fans around 32 and 64 sit on both sides of the pipelined path."""
    r, s0, c0 = 0, 1, 2
    g0, x0 = c0 + fan, c0 + 2 * fan
    src = [[r, s0], [r] * fan, np.arange(c0, g0)]
    dst = [[s0, r], np.arange(c0, g0), np.arange(g0, x0)]
    dense = 260
    a, b = np.meshgrid(np.arange(dense), np.arange(dense))
    n = x0 + dense
    src, dst = (np.concatenate(v + [x0 + z.ravel()]) for v, z in ((src, a), (dst, b)))
    _counts_equal(n, src, dst, [c0, g0, c0 + fan - 1], 0.3, budget)
