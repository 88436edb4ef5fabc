"""The pairwise Monte Carlo's flat loop: pair counts at the edges of a block, threads that take several walk pairs in
turn, walks of at most one and two nodes, equal nodes and nodes without in-neighbours; meet counts equal the oracle's."""
import numpy as np
import pytest

from gpu_util import gpu_graph, oracle_graph
from paper_1709_06955_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("npairs,r,lmax", [(1, 255, 64), (1, 256, 64), (1, 257, 64), (400, 9001, 64), (3, 700, 1),
                                           (3, 700, 2)])
def test_meets_equal_the_oracle(npairs, r, lmax):
    from paper_1709_06955_gb300 import build
    from oracle import build as obuild
    build.build()
    obuild.build()
    n, s, d = synth.config_graph("chunglu-1k")
    keep = d != 7  # node 7 has no in-neighbours
    s, d = s[keep], d[keep]
    G, O = gpu_graph(n, s, d, l_max=lmax), oracle_graph(n, s, d)
    rng = np.random.default_rng(npairs + r)
    us, vs = (rng.integers(0, n, npairs).astype(np.int32) for _ in range(2))
    if npairs > 2:
        us[0], vs[0], us[1] = 3, 3, 7
    ku, kv = np.arange(npairs, dtype=np.uint32), np.arange(npairs, dtype=np.uint32) + 9000
    meets, est = G.pair_mc(us, vs, ku, kv, r)
    for i in range(min(npairs, 40)):
        ref = O.pair_mc(int(us[i]), int(vs[i]), 0.6, lmax, 3, int(ku[i]), int(kv[i]), r)
        assert meets[i] == (r if us[i] == vs[i] else round(ref * r))
    G.close()
