"""Randomized calls over a level list that an earlier call left just large enough: two calls whose level 0 is sized to
exactly the kept capacity while the share of its items is no whole number of entries.  Exact member counts."""
import math

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


def level0_items(O, out_deg, u, qid, nr):
    """Work items of level 0: the out-degrees of every walk's nodes after the first."""
    return sum(int(out_deg[O.walk(u, 0.6, 64, 3, qid, k)[1:]].sum()) for k in range(nr))


def test_a_kept_list_of_exactly_the_size_wanted():
    from oracle import core
    from paper_1709_06955_gb300 import probesim
    n = 200
    s, d = dedup(n, *synth.chung_lu(n, 2000, seed=1))
    share = max(0.125, 4.0 * math.sqrt(0.6) * n / s.size)
    O, out_deg = oracle_graph(n, s, d), np.bincount(s, minlength=n)
    nr = core.num_walks(0.6, 0.3, 0.01, n)
    calls = [(170, 0), (167, 160)]
    first, second = [level0_items(O, out_deg, u, qid, nr) for u, qid in calls]
    sized = [int(share * e) + 1 for e in (first, second)]
    kept = (32 * sized[0] + 32 * sized[0] // 8) // 32  # the list a first call leaves, in entries of 32 bytes
    assert kept == sized[1] and int((kept - 1) / share) < second  # the second call's list is kept, with nothing to spare
    G = probesim.Graph(n, s, d, probe_mode=probesim.PROBE_RANDOMIZED)
    for u, qid in calls:
        got = G.single_source(probesim.make_queries([u], eps=0.3, query_ids=[qid]))[0]
        ref, _ = O.single_source(u, eps=0.3, seed=3, qid=qid, probe_mode=1)
        got, want = np.rint(got.astype(np.float64) * nr), np.rint(ref * nr)
        got[u] = want[u] = 0
        assert np.array_equal(got, want)
    G.close()
