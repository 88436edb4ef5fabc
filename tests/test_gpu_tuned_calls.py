"""A tuned graph's calls against the untuned ones': the tuner times the kernels that the level loop launches, so a tuned call
is no slower (beyond the timings' spread), and its scores are the same up to the order of sums."""
import time

import numpy as np
import pytest

from gpu_util import TOL, dedup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_06955_gb300 import build
    build.build()


def test_a_tuned_call_is_not_slower():
    """50,000 nodes and about 5 million edges: depths of hundreds of columns, pulled in 128-column tiles.  (Blocks per SM
    timed on one pair of 32-column tiles made a tuned call 8 to 9 % slower here.)"""
    import torch
    from paper_1709_06955_gb300 import probesim
    n, m = 50000, 5_500_000
    rng = np.random.default_rng(50)
    s = rng.permutation(n)[(n * rng.random(m) ** 3).astype(np.int64)]
    d = rng.permutation(n)[(n * rng.random(m) ** 2).astype(np.int64)]
    s, d = dedup(n, s, d)
    graphs = [probesim.Graph(n, s, d) for _ in range(2)]
    graphs[1].autotune()
    Q = probesim.make_queries(rng.choice(np.unique(d), 2, replace=False).tolist(), eps=0.1, query_ids=[1, 2])
    out = [torch.empty(2, n, device="cuda") for _ in graphs]
    best = [1e30, 1e30]
    for _ in range(24):
        for i, G in enumerate(graphs):
            torch.cuda.synchronize()
            t = time.perf_counter()
            G.single_source(Q, out=out[i])
            best[i] = min(best[i], time.perf_counter() - t)
    for G in graphs:
        G.close()
    assert float((out[0] - out[1]).abs().max()) <= TOL
    print("untuned %.3f ms, tuned %.3f ms" % (1e3 * best[0], 1e3 * best[1]))
    assert best[1] <= 1.05 * best[0]
