"""The frontier engine's task lists under a small memory budget.  Probes at their last level have tasks but neither a next
frontier nor a table, so the number of tasks alone must make the engine set probes aside; the estimates do not change."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_06955_gb300 import build
    build.build()


@pytest.mark.parametrize("cfg", [dict(eps_p=1e-6), dict(probe_mode=2, c0=1e30)])
def test_last_level_tasks_are_cut_by_the_budget(cfg):
    """Walks of at most two nodes on the complete graph of 1,000: every prefix is probed once, at its last level."""
    from paper_1709_06955_gb300 import probesim
    n, B, eps = 1000, 20, 0.3
    s, d = np.divmod(np.arange(n * n), n)
    s, d = s[s != d], d[s != d]
    G = probesim.Graph(n, s, d, l_max=2, **cfg)
    Q = probesim.make_queries(list(range(B)), eps=eps, query_ids=np.arange(B) + 5)
    want = G.single_source(Q)
    full = G.stats()
    assert full["deferred"] == 0 and full["levels"] == 1
    budget = 4 * 8 * 2 * B * G.num_walks(eps)  # the least that keeps the call in one batch
    assert full["probes"] > max(n, budget // 16 // 8)  # a task a probe: more than the budget's sixteenth
    G.set_memory_budget(budget)
    got, cut = G.single_source(Q), G.stats()
    G.close()
    assert cut["probes"] == full["probes"] and cut["edge_gathers"] == full["edge_gathers"]
    assert cut["deferred"] > 0
    assert np.array_equal(got, want)
