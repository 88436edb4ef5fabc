"""Top-k's candidate list against the full radix select (topk_select_noalloc, the same ranking over given scores): node
counts around the candidate capacity, ties that overflow it, k of 1 to 1,024 and above, few positive scores."""
import numpy as np
import pytest

from paper_1709_06955_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(40, 300), (4095, 30000), (4096, 30000), (4097, 30000), (9001, 20000), (60001, 900001)])
@pytest.mark.parametrize("mode", ["rand", "det"])
def test_equals_the_radix_select(n, m, mode):
    import torch
    from paper_1709_06955_gb300 import build, probesim
    build.build()
    s, d = synth.chung_lu(n, m, seed=n)
    G = probesim.Graph(n, s, d, probe_mode=probesim.PROBE_RANDOMIZED if mode == "rand" else 0)
    qs = synth.queries(n, d, 3, seed=1)
    for ks in ([1, 5, 39], [50, 1, 100], [1024, 1000, 7], [1500, 3, 1025]):
        ks = [min(k, n - 1) for k in ks]
        kmax = max(ks)
        Q = probesim.make_queries(qs, eps=0.3, k=ks, query_ids=[3, 4, 5])
        ids, vals = G.topk(Q, kmax=kmax)
        if mode == "det":  # the same scores only up to rounding: rank the call's own
            assert np.all(np.diff(vals, axis=1)[:, :1] <= 0)
            for i, k in enumerate(ks):
                order = np.lexsort((ids[i, :k], -vals[i, :k].astype(np.float64)))
                assert np.array_equal(order, np.arange(k)) and qs[i] not in ids[i, :k]
                assert np.all(ids[i, k:] == -1) and np.all(vals[i, k:] == 0) and np.unique(ids[i, :k]).size == k
            continue
        scores = torch.empty(3, n, device="cuda")
        G.single_source(Q, out=scores)
        if kmax <= 1024:
            ri = torch.empty(3, kmax, dtype=torch.int32, device="cuda")
            rv = torch.empty(3, kmax, device="cuda")
            probesim.topk_select_noalloc(scores, qs, ks, kmax, ri, rv)
            ri, rv = ri.cpu().numpy(), rv.cpu().numpy()
        else:
            sc = scores.cpu().numpy().astype(np.float64)
            ri, rv = np.full((3, kmax), -1, np.int32), np.zeros((3, kmax), np.float32)
            for i, k in enumerate(ks):
                sc[i, qs[i]] = -1
                top = np.lexsort((np.arange(n), -sc[i]))[:k]
                ri[i, :k], rv[i, :k] = top, sc[i, top]
        assert np.array_equal(ids, ri) and np.array_equal(vals, rv)
    G.close()
