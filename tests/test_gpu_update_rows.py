"""Update batches against a graph built from the edited edge list: walks (in-lists) and randomized estimates (out-lists)
are equal exactly.  Batches at the edges of the list copy: first and last rows, rows without entries, runs of touched
rows, one row taking a whole batch, batches larger than a copy tile, everything deleted."""
import numpy as np
import pytest

from gpu_util import dedup

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1709_06955_gb300 import build
    build.build()


def _same(G, n, keys, nodes):
    from paper_1709_06955_gb300 import probesim
    F = probesim.Graph(n, keys // n, keys % n, probe_mode=probesim.PROBE_RANDOMIZED)
    Q = probesim.make_queries(nodes, eps=0.3, query_ids=np.arange(len(nodes)))
    assert G.info()[1] == F.info()[1]
    for a, b in zip(G.sample_walks(Q), F.sample_walks(Q)):
        assert np.array_equal(a, b)
    assert np.array_equal(G.single_source(Q), F.single_source(Q))
    F.close()


def _batches(n, rng):
    every = np.arange(n)
    yield np.array([0, n - 1, n - 1]), np.array([n - 1, 0, 1])            # first and last rows
    yield np.full(n - 1, 0), every[1:]                                    # one out-list, every in-list
    yield every[1:], np.full(n - 1, 0)                                    # one in-list, every out-list
    yield every[:-1][n // 3:2 * n // 3], every[1:][n // 3:2 * n // 3]     # a run of neighbouring rows
    yield rng.integers(0, n, 5 * n), rng.integers(0, n, 5 * n)            # loops, repeats, edges that exist
    yield np.array([5, 5]), np.array([5, 5])                              # nothing


@pytest.mark.parametrize("n,m", [(33, 60), (700, 2047), (700, 2049), (5000, 70001)])
def test_batches_equal_a_fresh_build(n, m):
    from paper_1709_06955_gb300 import probesim
    rng = np.random.default_rng(n + m)
    s, d = rng.integers(0, n, m), rng.integers(0, n, m)
    s[s % 7 == 3] = 1  # rows without out-edges, and a hub
    d[d % 5 == 2] = 2
    s, d = dedup(n, s, d)
    keys = np.unique(s.astype(np.int64) * n + d)
    G = probesim.Graph(n, s, d, probe_mode=probesim.PROBE_RANDOMIZED)
    nodes = [0, 2, n - 1, int(rng.integers(n))]
    for bs, bd in _batches(n, rng):
        bk = np.unique((bs.astype(np.int64) * n + bd)[bs != bd])
        new = np.union1d(keys, bk)
        assert G.insert_edges(bs, bd) == new.size - keys.size
        keys = new
        _same(G, n, keys, nodes)
        drop = np.concatenate([rng.choice(keys, keys.size // 3, replace=False), bk[::2]])
        new = np.setdiff1d(keys, drop)
        assert G.delete_edges(drop // n, drop % n) == keys.size - new.size
        keys = new
        _same(G, n, keys, nodes)
    assert G.delete_edges(keys // n, keys % n) == keys.size
    assert G.info()[1] == 0
    assert G.insert_edges([1, 2, 3], [0, 1, 0]) == 3
    _same(G, n, np.array([n, 2 * n + 1, 3 * n], np.int64), nodes)
    G.close()


@pytest.mark.parametrize("memory", ["device", "pinned", "host"])
def test_update_reads_edges_that_the_callers_stream_writes(memory):
    """A batch runs on the graph's own stream; edges in device or pinned memory are read after the work that the caller's
    stream already holds, here products of two matrices and then the copies that write the edges."""
    import torch
    from paper_1709_06955_gb300 import probesim
    n, rng = 3000, np.random.default_rng(12)
    s, d = dedup(n, rng.integers(0, n, 20000), rng.integers(0, n, 20000))
    keys = np.unique(s.astype(np.int64) * n + d)
    es, ed = (rng.integers(0, n, 4000).astype(np.int32) for _ in range(2))
    G = probesim.Graph(n, keys // n, keys % n, probe_mode=probesim.PROBE_RANDOMIZED)
    stream = torch.cuda.Stream()
    a = torch.randn(4096, 4096, device="cuda")
    bufs = [torch.zeros(4000, dtype=torch.int32, device="cuda" if memory == "device" else "cpu",
                        pin_memory=memory == "pinned") for _ in range(2)]
    from_dev = [torch.tensor(x, device="cuda") for x in (es, ed)]
    torch.cuda.synchronize()
    with torch.cuda.stream(stream):
        for _ in range(30):
            a = (a @ a) * 1e-3
        for b, f in zip(bufs, from_dev):
            b.copy_(f, non_blocking=memory != "host")
    args = bufs if memory == "device" else [b.numpy() for b in bufs]
    G.insert_edges(args[0], args[1], stream=stream.cuda_stream)
    torch.cuda.synchronize()
    added = (es.astype(np.int64) * n + ed)[es != ed]
    _same(G, n, np.union1d(keys, added), [1, 2, 3])
    G.close()
