"""Deterministic calls on several graphs from several threads at once.  The accumulate stages rows of as many columns as a
call's walk tree needs, in as much shared memory; calls of very different widths must not disturb each other."""
import threading

import numpy as np
import pytest

from paper_1709_06955_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_06955_gb300 import build
    build.build()


def test_calls_of_different_widths_at_once():
    from paper_1709_06955_gb300 import probesim
    jobs = []
    for n, m, eps in [(900, 20000, 0.05), (1000, 30000, 0.05), (800, 6000, 0.3), (1100, 30000, 0.1)]:
        s, d = synth.chung_lu(n, m, seed=n)
        G = probesim.Graph(n, s, d)
        u = int(synth.queries(n, d, 1, seed=1)[0])
        Q = probesim.make_queries([u], eps=eps, query_ids=[n])
        alone = [G.single_source(Q)[0] for _ in range(2)]
        jobs.append((G, Q, alone, G.stats()["max_columns"]))
    cols = sorted(j[3] for j in jobs)
    # rows of the same staging class (8 a block: at most 3,584 columns), some above the 48 KB (1,536 columns) a kernel gets
    # without asking
    assert cols[0] < 1536 and any(1536 < c <= 3584 for c in cols)
    stop, errors = threading.Event(), []

    def run(G, Q, alone, _):
        try:
            for _ in range(150):
                if stop.is_set():
                    return
                got = G.single_source(Q)[0]
                np.testing.assert_allclose(got, alone[0], rtol=0, atol=2e-6)
        except Exception as e:  # a failed launch, or other scores
            errors.append(repr(e)[:300])
            stop.set()

    threads = [threading.Thread(target=run, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for G, *_ in jobs:
        G.close()
    assert not errors
