"""The level loop's pull tiles: narrow tails by eight lanes a piece, 128-column tiles with up to three 32-column tiles
after them, in the node-major and the grouped layout, on both sides of the rules that choose them, against the oracle."""
import numpy as np
import pytest

from gpu_util import TOL, dedup, gpu_graph, oracle_graph
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


def _check(n, s, d, nq, eps, walks):
    from paper_1709_06955_gb300 import probesim
    s, d = dedup(n, s, d)
    G, O = gpu_graph(n, s, d), oracle_graph(n, s, d)
    qs = synth.queries(n, d, nq, seed=nq)
    Q = probesim.make_queries(qs, eps=eps, query_ids=np.arange(nq) + 9, walk_begin=0, walk_end=walks)
    out = G.single_source(Q)
    cols = G.stats()["max_columns"]
    G.close()
    for t in {0, nq - 1}:
        ref, _ = O.single_source(int(qs[t]), eps=eps, seed=3, qid=9 + t, walk_begin=0, walk_end=walks)
        assert np.max(np.abs(out[t] - ref)) <= TOL
    return cols


@pytest.mark.parametrize("nq,walks", [(1, 3), (1, 9), (1, 20), (1, 150), (1, 400), (2, 400), (1, 1000), (3, 900),
                                      (5, 1000), (9, 1000)])
def test_widths_from_one_column_to_several_groups(nq, walks):
    """11,000 rows: wide tiles from 128 columns on once there are two of them."""
    n = 11003
    s, d = synth.chung_lu(n, 100000, seed=3)
    _check(n, s, d, nq, 0.15, walks)


def test_tiny_and_split_rows():
    """Rows cut into pieces (in-degree above 128) through the narrow tails' atomic adds; fewer rows than a warp."""
    for n in (17, 700):
        rng = np.random.default_rng(n)
        s, d = rng.integers(0, n, 40 * n), rng.integers(0, n, 40 * n)
        d[: n // 2] = 0
        s[: n // 2] = np.arange(n // 2) + 1
        _check(n, s, d, 2, 0.2, 300)


def test_more_pieces_than_the_narrow_rule():
    n, s, d = synth.rmat(18, 1 << 20, seed=2)
    _check(n, s, d, 1, 0.2, 12)
