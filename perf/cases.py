"""Performance cases of the ProbeSim library: the calls a user's program makes, over the sizes it makes them at.

Each case is a dict of plain values.  Its ``kind`` says which public call it times:

  single_source  ``Graph.single_source``: the estimates of every node for a call's queries
  topk           ``Graph.topk``: top-k lists
  serve          a burst of top-k queries through the continuous-batching ``Server``
  update         a batch of edge insertions, a query on the new graph, and the batch deleted again
  build          ``Graph(...)`` from an edge list on the device, and a first short query on it
  pair_mc        ``Graph.pair_mc``: single-pair Monte Carlo estimates

and ``mode`` the PROBE variant: ``det`` (Alg. 2), ``rule2`` (Alg. 2 with Thm. 2's split of the error over both pruning
rules), ``switch`` (Sec. 4.4, c0 = 0.01) or ``rand`` (Alg. 3).  Graphs are R-MAT (.57, .19, .19, .05) or Chung-Lu
(exponent 2.1), drawn on the GPU from the seed alone; query nodes are uniform over the nodes with an in-neighbour.

Deterministic PROBE returns whole score rows; the top-k lists come from the modes whose sums are exact integers, so
their ids are the same in every run.  ``exact`` replays a call's Philox walks and evaluates Algs. 1-4 in FP64 with
plain torch operations.
"""
import math

import numpy as np
import torch

from paper_1709_06955_gb300 import probesim

C_DECAY, DELTA, SEED, L_MAX = 0.6, 0.01, 3, 64
MODES = {"det": probesim.PROBE_DETERMINISTIC, "rule2": probesim.PROBE_DETERMINISTIC,
         "rand": probesim.PROBE_RANDOMIZED, "switch": probesim.PROBE_SWITCH}


def listed():
    def case(name, kind, mode, graph, n, m, nq, eps, **kw):
        d = {"name": name, "kind": kind, "mode": mode, "graph": graph, "n": n, "m": m, "nq": nq, "eps": eps,
             "k": "50", "host_out": False, "batch": 0, "pairs": 0, "r": 0}
        d.update(kw)
        return d

    return [
        # the paper's small-graph study: one interactive query on a graph of 1,000 nodes; launches and latency
        case("ss_tiny", "single_source", "det", "chung_lu", 1000, 10000, 1, "0.1"),
        # a small call at odd sizes, uneven accuracy, scores returned to host memory
        case("ss_ragged_host", "single_source", "det", "chung_lu", 30011, 400003, 3, "0.1,0.15", host_out=True),
        # the headline: one query at a time on a graph of a million nodes, scores kept on the device
        case("ss_rmat20", "single_source", "det", "rmat", 1 << 20, 1 << 24, 1, "0.1"),
        # a batch at high accuracy on a mid-sized graph (four times the walks of the headline's queries)
        case("ss_rmat18_fine", "single_source", "det", "rmat", 1 << 18, 1 << 22, 2, "0.05"),
        # Thm. 2's guaranteed error 0.1 with both pruning rules and the estimate shift, off a power of two
        case("ss_rule2", "single_source", "rule2", "rmat", 150001, 2400007, 1, "0.1"),
        # randomized PROBE: a small batch of top-k queries
        case("topk_rand20", "topk", "rand", "rmat", 1 << 20, 1 << 24, 4, "0.1"),
        # the switch of Sec. 4.4: one interactive top-k query
        case("topk_switch20_one", "topk", "switch", "rmat", 1 << 20, 1 << 24, 1, "0.1"),
        # the batched configuration: many queries with uneven accuracy in one call on a graph of 67 million edges
        case("topk_switch22_batch", "topk", "switch", "rmat", 1 << 22, 1 << 26, 64, "0.1,0.05"),
        # the serving configuration: a burst of requests with uneven accuracy and k
        case("serve_burst20", "serve", "switch", "rmat", 1 << 20, 1 << 24, 12, "0.1,0.05,0.025", k="10,50,100"),
        # dynamic graph: 10,000 insertions, a query, 10,000 deletions
        case("update_10k", "update", "switch", "rmat", 1 << 21, 1 << 25, 1, "0.1", batch=10000),
        # a graph taken in: an odd-sized edge list on the device to a first answer
        case("build_odd", "build", "rand", "rmat", 700001, 11000003, 1, "0.1"),
        # the single-pair estimator gauging pooled candidates
        case("pair_mc20", "pair_mc", "det", "rmat", 1 << 20, 1 << 24, 0, "0.1", pairs=50, r=1 << 20),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["single_source"] * 4 + ["topk"] * 4 + ["serve", "update", "build", "pair_mc"])
    mode = {"single_source": ["det", "det", "det", "rule2"], "topk": ["rand", "switch", "switch"],
            "serve": ["switch"], "update": ["switch"], "build": ["rand"], "pair_mc": ["det"]}[kind]
    mode = rng.choice(mode)
    hi = {"single_source": 1 << 20, "topk": 1 << 22, "serve": 1 << 20, "update": 1 << 22, "build": 1 << 22,
          "pair_mc": 1 << 22}[kind]
    if mode == "rule2":
        hi = 150001
    n = _log(rng, 1000 if kind == "single_source" else 20000, hi)
    if rng.random() < 0.25:
        n = min(hi, 1 << max(10, n.bit_length() - 1))
    m = int(n * rng.uniform(8.0, 16.0))
    graph = "chung_lu" if n <= 60000 and rng.random() < 0.5 else "rmat"
    # a call of the deterministic modes stays within the walks x edges of the largest listed ones
    if kind == "single_source":
        eps = "0.1" if mode == "rule2" else rng.choice(["0.1", "0.15", "0.1,0.05"] if n <= 300000 else ["0.1", "0.15"])
        nq = 1 if mode == "rule2" else rng.randint(1, max(1, min(8, (3 << 20) // n)))
    elif kind == "topk":
        eps = rng.choice(["0.1", "0.1,0.05", "0.05"])
        nq = rng.randint(1, max(1, min(64, (32 << 20) // n)))
    elif kind == "serve":
        eps, nq = rng.choice(["0.1,0.05", "0.1,0.05,0.025"]), rng.randint(2, 12)
    else:
        eps, nq = "0.1", 0 if kind == "pair_mc" else 1
    return {"kind": kind, "mode": mode, "graph": graph, "n": n, "m": m, "nq": nq, "eps": eps,
            "k": rng.choice(["10", "50", "100", "10,50,100"]), "host_out": bool(rng.random() < 0.3),
            "batch": _log(rng, 100, 20000) if kind == "update" else 0,
            "pairs": rng.randint(1, 50) if kind == "pair_mc" else 0,
            "r": _log(rng, 10000, 1 << 20) if kind == "pair_mc" else 0}


# ---------------------------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _draw_edges(case, k, gen, state):
    """k candidate edges (src, dst) as int64."""
    n = case["n"]
    if case["graph"] == "rmat":
        bits = (n - 1).bit_length()
        src = torch.zeros(k, dtype=torch.int64, device="cuda")
        dst = torch.zeros(k, dtype=torch.int64, device="cuda")
        for b in range(bits):
            r = torch.rand(k, generator=gen, device="cuda")
            src |= (r >= 0.76).long() << b
            dst |= (((r >= 0.57) & (r < 0.76)) | (r >= 0.95)).long() << b
        ok = (src < n) & (dst < n) & (src != dst)
        return src[ok], dst[ok]
    if "cdf" not in state:
        w = (torch.arange(n, device="cuda", dtype=torch.float64) + 1.0) ** (-1.0 / 1.1)
        state["cdf"] = [torch.cumsum(w[torch.randperm(n, generator=gen, device="cuda")], 0) for _ in range(2)]
    out = []
    for cdf in state["cdf"]:
        u = torch.rand(k, generator=gen, device="cuda", dtype=torch.float64) * cdf[-1]
        out.append(torch.searchsorted(cdf, u).clamp_(max=n - 1))
    ok = out[0] != out[1]
    return out[0][ok], out[1][ok]


def _edges(case, seed):
    """m distinct loop-free edges in random order with random node labels: int32 (src, dst) on the GPU."""
    n, m = case["n"], case["m"]
    gen, state = _gen(seed), {}
    keys = torch.empty(0, dtype=torch.int64, device="cuda")
    while keys.numel() < m:
        s, d = _draw_edges(case, max(4096, int((m - keys.numel()) * 1.3)), gen, state)
        keys = torch.unique(torch.cat([keys, s * n + d]))
    keys = keys[torch.randperm(keys.numel(), generator=gen, device="cuda")[:m]]
    label = torch.randperm(n, generator=gen, device="cuda")
    return label[keys // n].int(), label[keys % n].int()


def _floats(text):
    return [float(x) for x in text.split(",")]


def _query_args(case, seed, dst):
    """Query nodes, accuracies, list lengths and Philox ids of the case's queries."""
    nq = max(1, case["nq"])
    rng = np.random.default_rng(seed + 17)
    cand = np.nonzero(torch.bincount(dst.long(), minlength=case["n"]).cpu().numpy() > 0)[0]
    nodes = rng.choice(cand, size=nq, replace=nq > cand.size).astype(np.int32)
    eps, ks = _floats(case["eps"]), [int(x) for x in case["k"].split(",")]
    return (nodes, [eps[i % len(eps)] for i in range(nq)], [ks[i % len(ks)] for i in range(nq)],
            (np.arange(nq) + 1000 * (seed % 1000)).astype(np.int64))


def _config(case):
    kw = {"c": C_DECAY, "delta": DELTA, "l_max": L_MAX, "seed": SEED, "probe_mode": MODES[case["mode"]]}
    if case["mode"] == "switch":
        kw["c0"] = 0.01
    if case["mode"] == "rule2":
        sp = probesim.split_error(_floats(case["eps"])[0], C_DECAY, True)
        kw.update(l_max=sp["l_max"], eps_p=sp["eps_p"], shift=sp["shift"])
    return kw


def _batch(case, seed, src, dst):
    """An update batch: mostly new random edges, some that exist already (skipped by the call)."""
    gen = _gen(seed + 29)
    k, n = case["batch"], case["n"]
    s = torch.randint(0, n, (k,), generator=gen, device="cuda", dtype=torch.int32)
    d = torch.randint(0, n, (k,), generator=gen, device="cuda", dtype=torch.int32)
    # sources follow the graph's own out-degrees for every other edge, as attachments do
    e = torch.randint(0, case["m"], ((k + 1) // 2,), generator=gen, device="cuda")
    s[::2] = src[e]
    keys = torch.unique(src.long() * n + dst.long())
    new = s.long() * n + d.long()
    at = torch.searchsorted(keys, new).clamp_(max=keys.numel() - 1)
    fresh = keys[at] != new  # an edge that exists would be deleted with the batch: the graph must come back as it was
    return s[fresh].cpu().numpy(), d[fresh].cpu().numpy()


def prepare(case, seed):
    src, dst = _edges(case, seed)
    kind = case["kind"]
    st = {"case": case}
    nodes, eps, ks, qid = _query_args(case, seed, dst)
    if case["mode"] == "rule2":
        eps = [probesim.split_error(e, C_DECAY, True)["eps"] for e in eps]
    if kind == "build":
        st.update(src=src, dst=dst, config=_config(case), out=torch.empty(1, case["n"], device="cuda"),
                  queries=probesim.make_queries(nodes, eps=eps, k=ks, query_ids=qid, walk_begin=0, walk_end=64))
        return st
    st["graph"] = probesim.Graph(case["n"], src, dst, **_config(case))
    st["queries"] = probesim.make_queries(nodes, eps=eps, k=ks, query_ids=qid)
    if kind in ("single_source", "update"):
        st["out"] = (np.empty((len(nodes), case["n"]), np.float32) if case["host_out"]
                     else torch.empty(len(nodes), case["n"], device="cuda"))
    if kind == "update":
        st["batch"] = _batch(case, seed, src, dst)
    elif kind == "serve":
        st["server"] = probesim.Server(st["graph"], workers=3, max_batch=2, kmax=100)
    elif kind == "pair_mc":
        st["pairs"] = _pairs(case, seed)
    return st


def _pairs(case, seed):
    rng = np.random.default_rng(seed + 5)
    u = np.full(case["pairs"], rng.integers(case["n"]), np.int32)  # one pooled node against its candidates
    v = rng.integers(0, case["n"], case["pairs"]).astype(np.int32)
    return u, v, np.full(case["pairs"], 1, np.uint32), (np.arange(case["pairs"]) + 2).astype(np.uint32)


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "single_source":
        return state["graph"].single_source(state["queries"], out=state["out"])
    if kind == "topk":
        return state["graph"].topk(state["queries"])
    if kind == "update":
        g = state["graph"]
        added = g.insert_edges(*state["batch"])
        scores = g.single_source(state["queries"], out=state["out"])
        return [added, scores, g.delete_edges(*state["batch"])]
    if kind == "build":
        g = probesim.Graph(case["n"], state["src"], state["dst"], **state["config"])
        n, m, _ = g.info()
        nodes, lens = g.sample_walks(state["queries"])
        scores = g.single_source(state["queries"], out=state["out"])
        g.close()
        return [n, m, nodes, lens, scores]
    if kind == "pair_mc":
        return state["graph"].pair_mc(*state["pairs"], case["r"])
    tickets = state["server"].submit(state["queries"])
    done = {}
    while len(done) < len(tickets):
        for res, ids, vals in state["server"].poll(max_results=64, wait_ms=100):
            done[res.ticket] = (ids, vals)
    return [np.stack([done[t][0] for t in tickets]), np.stack([done[t][1] for t in tickets])]


# ---------------------------------------------------------------------------------------------------------------
# work
# ---------------------------------------------------------------------------------------------------------------
def _num_walks(case, eps):
    return math.ceil(3.0 * C_DECAY / (eps * eps) * math.log(case["n"] / DELTA))


def work(case):
    """Bytes: the adjacency the path reads (each list once) and the outputs.  Operations: for the deterministic PROBE
    one multiply and add per edge and level of the deepest walk (a product with the transition matrix per level); for
    the sampled paths about 100 integer operations per walk step (a ten-round Philox block and the step)."""
    n, m, nq = case["n"], case["m"], max(1, case["nq"])
    lists = 4.0 * m + 8.0 * (n + 1)
    eps = _floats(case["eps"])
    if case["mode"] == "rule2":
        eps = [e / 2.0 for e in eps]
    walks = [_num_walks(case, eps[i % len(eps)]) for i in range(nq)]
    steps = 4.4 * sum(walks)
    levels = sum(math.log(w) / -math.log(math.sqrt(C_DECAY)) for w in walks)
    kind = case["kind"]
    if kind == "pair_mc":
        return {"bytes": lists + 12.0 * case["pairs"], "flops": 2.0 * 2.5 * 100.0 * case["pairs"] * case["r"]}
    if kind == "build":
        return {"bytes": 8.0 * m + 2.0 * lists + 4.0 * n, "flops": 4.0 * m}
    if kind == "update":  # both lists read and written by each of the two batches, and one query's scores
        return {"bytes": 2.0 * 2.0 * 2.0 * lists + 4.0 * n, "flops": 100.0 * steps}
    out = 4.0 * n * nq if kind == "single_source" else 8.0 * 100 * nq
    if case["mode"] == "det":
        return {"bytes": lists + out, "flops": 2.0 * m * levels}
    return {"bytes": 2.0 * lists + out, "flops": 100.0 * steps}


# ---------------------------------------------------------------------------------------------------------------
# exact: Algs. 1-4 in FP64, from the inputs alone
# ---------------------------------------------------------------------------------------------------------------
_U32 = 0xFFFFFFFF
T_STOP = int(math.floor((1.0 - math.sqrt(C_DECAY)) * 4294967296.0))
T_KEEP = int(math.floor(math.sqrt(C_DECAY) * 4294967296.0))


def _philox(c0, c1, c2, k0, k1):
    """Philox4x32-10 of counter (c0, c1, c2, 0) under key (k0, k1): words 0 and 1, on int64 tensors of uint32 values."""
    c3 = torch.zeros_like(c0)
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & _U32, (k1 + 0xBB67AE85) & _U32
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # wraps; the shifts below take the unsigned halves
        c0, c1, c2, c3 = ((p1 >> 32) & _U32) ^ c1 ^ k0, p1 & _U32, ((p0 >> 32) & _U32) ^ c3 ^ k1, p0 & _U32
    return c0, c1


def _mulhi(a, b):
    return ((a * b) >> 32) & _U32


class _Lists:
    """In-lists in source order and out-lists, as offsets and columns (int64)."""

    def __init__(self, n, src, dst):
        self.n = n
        src, dst = src.long(), dst.long()
        key = torch.sort(dst * n + src)[0]
        self.in_col, v = key % n, key // n
        self.deg_in = torch.bincount(v, minlength=n)
        self.in_off = torch.cumsum(self.deg_in, 0) - self.deg_in
        key = torch.sort(src * n + dst)[0]
        self.out_col = key % n
        self.deg_out = torch.bincount(key // n, minlength=n)
        self.out_off = torch.cumsum(self.deg_out, 0) - self.deg_out
        self.w = math.sqrt(C_DECAY) / self.deg_in.clamp(min=1).double()

    def walks(self, u, eps_walks, qid, l_max, count=None):
        W = eps_walks if count is None else min(count, eps_walks)
        k = torch.arange(W, device="cuda")
        nodes = torch.full((W, l_max), -1, dtype=torch.int64, device="cuda")
        nodes[:, 0] = u
        lens = torch.ones(W, dtype=torch.int64, device="cuda")
        live, v = k, torch.full((W,), u, dtype=torch.int64, device="cuda")
        for s in range(l_max - 1):
            x0, x1 = _philox(live, torch.full_like(live, s), torch.zeros_like(live), SEED, torch.full_like(live, qid))
            go = (x0 >= T_STOP) & (self.deg_in[v] > 0)
            live, v, x1 = live[go], v[go], x1[go]
            if live.numel() == 0:
                break
            v = self.in_col[self.in_off[v] + _mulhi(x1, self.deg_in[v])]
            nodes[live, s + 1] = v
            lens[live] += 1
        return nodes, lens

    def expand(self, nodes):
        """Out-edges of the nodes: (index into nodes, destination)."""
        d = self.deg_out[nodes]
        row = torch.repeat_interleave(torch.arange(nodes.numel(), device="cuda"), d)
        first = torch.cumsum(d, 0) - d
        return row, self.out_col[self.out_off[nodes][row] + torch.arange(row.numel(), device="cuda") - first[row]]


def _tree(n, nodes, lens):
    """The prefixes of the walks per depth d (1-based): (graph node, parent, weight), and each walk's prefix ids."""
    W, dmax = nodes.shape[0], int(lens.max())
    pid = torch.zeros(W, dtype=torch.int64, device="cuda")
    levels = [(nodes[:1, 0], torch.zeros(1, dtype=torch.int64, device="cuda"), torch.tensor([W], device="cuda"))]
    ids = torch.zeros(W, dmax, dtype=torch.int64, device="cuda")
    for d in range(2, dmax + 1):
        live = torch.nonzero(lens >= d)[:, 0]
        key, inv, cnt = torch.unique(pid[live] * n + nodes[live, d - 1], return_inverse=True, return_counts=True)
        pid[live] = inv
        ids[live, d - 1] = inv
        levels.append((key % n, key // n, cnt))
    return levels, ids


def _det_row(G, M, levels, n_r):
    """Horner's rule over the tree: C(t) = sum over children s of w_s/n_r e_{a_s} + X_{a_s} M C(s)."""
    n = G.n
    below = None  # (C matrix [n, number of owners], owner prefix ids) of the current depth
    for d in range(len(levels), 1, -1):
        a, parent, cnt = levels[d - 1]
        owners, col = torch.unique(parent, return_inverse=True)
        C = torch.zeros(n, owners.numel(), dtype=torch.float64, device="cuda")
        if below is not None:
            B, who = below
            for c0 in range(0, who.numel(), 256):  # the children's products, a block of columns at a time
                part = who[c0:c0 + 256]
                Y = torch.sparse.mm(M, B[:, c0:c0 + 256].contiguous())
                Y[a[part], torch.arange(part.numel(), device="cuda")] = 0.0
                C.index_add_(1, col[part], Y)
            del B
        C.view(-1).index_add_(0, a * owners.numel() + col, cnt.double() / n_r)
        below = (C, owners)
    if below is None:
        return torch.zeros(n, dtype=torch.float64, device="cuda")
    return torch.sparse.mm(M, below[0])[:, 0]


def _rand_counts(G, nodes, lens, qid, walk, plen, counts):
    """Alg. 3 for the instances (walk, prefix length): adds the members of the last level's set into counts."""
    n = G.n
    inst, y = torch.arange(walk.numel(), device="cuda"), nodes[walk, plen - 1]
    j = 0
    while inst.numel():
        on = plen[inst] - 2 >= j
        inst, y = inst[on], y[on]
        members = torch.sort(inst * n + y)[0]
        row, x = G.expand(y)
        it = inst[row]
        cand = torch.unique(it * n + x)
        it, x = cand // n, cand % n
        ok = x != nodes[walk[it], plen[it] - j - 2]
        it, x = it[ok], x[ok]
        if it.numel() == 0:
            break
        r0, r1 = _philox(walk[it], (1 << 24) | (plen[it] << 8) | j, x, SEED, torch.full_like(x, qid))
        ok = r1 < T_KEEP
        it, x, r0 = it[ok], x[ok], r0[ok]
        key = it * n + G.in_col[G.in_off[x] + _mulhi(r0, G.deg_in[x])]
        ok = members[torch.searchsorted(members, key).clamp_(max=members.numel() - 1)] == key
        it, x = it[ok], x[ok]
        last = plen[it] - 2 == j
        counts += torch.bincount(x[last], minlength=n)
        inst, y = it[~last], x[~last]
        j += 1


def _frontier_row(G, nodes, lens, qid, n_r, switch, c0, eps_p):
    """Every prefix probed on its own (Alg. 2 with Pruning Rule 2; with `switch`, Sec. 4.4)."""
    n = G.n
    levels, ids = _tree(n, nodes, lens)
    est = torch.zeros(n, dtype=torch.float64, device="cuda")
    counts = torch.zeros(n, dtype=torch.int64, device="cuda")
    for q in range(2, len(levels) + 1):
        a, _, cnt = levels[q - 1]
        path = torch.empty(a.numel(), q, dtype=torch.int64, device="cuda")  # a walk through each prefix
        live = torch.nonzero(lens >= q)[:, 0]
        path[ids[live, q - 1]] = nodes[live, :q]
        pr, x = torch.arange(a.numel(), device="cuda"), a.clone()
        sc = torch.ones(a.numel(), dtype=torch.float64, device="cuda")
        gone = torch.zeros(a.numel(), dtype=torch.bool, device="cuda")
        for j in range(q - 1):
            if eps_p > 0:
                ok = sc * math.sqrt(C_DECAY) ** (q - j - 1) > eps_p
                pr, x, sc = pr[ok], x[ok], sc[ok]
            if switch:
                total = torch.zeros_like(cnt).index_add_(0, pr, G.deg_out[x])
                gone |= total > torch.floor(c0 * cnt.double() * n).long()
                ok = ~gone[pr]
                pr, x, sc = pr[ok], x[ok], sc[ok]
            if pr.numel() == 0:
                break
            row, v = G.expand(x)
            p, val = pr[row], G.w[v] * sc[row]
            ok = v != path[p, q - j - 2]
            key, inv = torch.unique(p[ok] * n + v[ok], return_inverse=True)
            sc = torch.zeros(key.numel(), dtype=torch.float64, device="cuda").index_add_(0, inv, val[ok])
            pr, x = key // n, key % n
        if pr.numel():
            est.index_add_(0, x, sc * cnt[pr].double())
        if switch:
            w = live[gone[ids[live, q - 1]]]
            if w.numel():
                _rand_counts(G, nodes, lens, qid, w, torch.full_like(w, q), counts)
    return (est + counts.double()) / n_r


def _rows(case, src, dst, args, walk_count=None):
    """The estimates of the case's queries, [nq, n] in FP64."""
    n, mode = case["n"], case["mode"]
    nodes_q, eps, _, qid = args
    l_max, eps_p, shift = L_MAX, 0.0, 0.0
    if mode == "rule2":  # Thm. 2's split: half to sampling, a quarter to each pruning rule, Rule 1's part centred
        e, sc = eps[0], math.sqrt(C_DECAY)
        eps = [x / 2.0 for x in eps]
        eps_t = e / 2.0
        l_max = max(1, math.ceil(math.log(eps_t) / math.log(sc)))
        p = e / 4.0 / ((1.0 + e / 2.0) * sc / ((1.0 - sc) * (1.0 - sc)))
        f = np.float32(p)
        eps_p = float(np.nextafter(f, np.float32(0)) if float(f) > p else f)
        shift = float(np.float32(eps_t / 2.0))
    G = _Lists(n, src, dst)
    M = None
    if mode == "det":
        off = torch.cat([G.in_off, torch.tensor([G.in_col.numel()], device="cuda")])
        M = torch.sparse_csr_tensor(off, G.in_col, torch.repeat_interleave(G.w, G.deg_in), size=(n, n))
    out = torch.empty(len(nodes_q), n, dtype=torch.float64, device="cuda")
    for i, u in enumerate(nodes_q):
        n_r = _num_walks(case, eps[i])
        nodes, lens = G.walks(int(u), n_r, int(qid[i]), l_max, walk_count)
        if mode == "det":
            out[i] = _det_row(G, M, _tree(n, nodes, lens)[0], n_r)
        elif mode == "rand":
            counts = torch.zeros(n, dtype=torch.int64, device="cuda")
            for w0 in range(0, nodes.shape[0], 1024):  # walks a block at a time: the candidate sets are large
                blk = torch.arange(w0, min(w0 + 1024, nodes.shape[0]), device="cuda")
                probes = (lens[blk] - 1).clamp(min=0)
                w = torch.repeat_interleave(blk, probes)
                first = torch.cumsum(probes, 0) - probes
                plen = torch.arange(w.numel(), device="cuda") - torch.repeat_interleave(first, probes) + 2
                _rand_counts(G, nodes, lens, int(qid[i]), w, plen, counts)
            out[i] = counts.double() / n_r
        else:
            out[i] = _frontier_row(G, nodes, lens, int(qid[i]), n_r, mode == "switch", float(np.float32(0.01)), eps_p)
        out[i] += shift
        out[i, int(u)] = 1.0
    return out


def exact(case, seed):
    kind, n, m = case["kind"], case["n"], case["m"]
    src, dst = _edges(case, seed)
    if kind == "pair_mc":
        if case["pairs"] * case["r"] > 1 << 26:
            return None
        G = _Lists(n, src, dst)
        meets = [_pair_meets(G, *(int(z[i]) for z in _pairs(case, seed)), case["r"]) for i in range(case["pairs"])]
        return [np.array(meets, np.int64), np.array(meets, np.float64) / case["r"]]
    args = _query_args(case, seed, dst)
    if kind == "build":
        G = _Lists(n, src, dst)
        n_r = _num_walks(case, args[1][0])
        nodes, lens = G.walks(int(args[0][0]), n_r, int(args[3][0]), L_MAX, 64)
        rows = _rows(case, src, dst, args, 64)
        return [n, m, nodes.int().cpu().numpy(), lens.int().cpu().numpy(), rows]
    cost = m * sum(_num_walks(case, e) for e in args[1])  # edges x walks
    if cost > (8 << 36 if case["mode"] == "det" else 4 << 36):
        return None
    if kind == "update":
        s, d = (torch.from_numpy(z).cuda() for z in _batch(case, seed, src, dst))
        ok = s != d
        key = torch.unique(s[ok].long() * n + d[ok].long())
        rows = _rows(case, torch.cat([src.long(), key // n]), torch.cat([dst.long(), key % n]), args)
        return [int(key.numel()), rows, int(key.numel())]
    rows = _rows(case, src, dst, args)
    if kind == "single_source":
        return rows
    kmax = 100 if kind == "serve" else max(args[2])
    vals = torch.zeros(len(args[0]), kmax, dtype=torch.float64)
    for i, u in enumerate(args[0]):
        rows[i, int(u)] = -1.0
        vals[i, :args[2][i]] = torch.sort(rows[i], descending=True)[0][:args[2][i]].cpu()
    return [None, vals]


def _pair_meets(G, u, v, ku, kv, r):
    """Walk pairs (u, v) that meet, by lockstep."""
    if u == v:
        return r
    met = 0
    for t0 in range(0, r, 1 << 22):
        t = torch.arange(t0, min(r, t0 + (1 << 22)), device="cuda")
        a, b = torch.full_like(t, u), torch.full_like(t, v)
        for s in range(L_MAX - 1):
            step = torch.full_like(t, s)
            zero = torch.zeros_like(t)
            a0, a1 = _philox(t, step, zero, SEED, torch.full_like(t, ku))
            b0, b1 = _philox(t, step, zero, SEED, torch.full_like(t, kv))
            go = (a0 >= T_STOP) & (b0 >= T_STOP) & (G.deg_in[a] > 0) & (G.deg_in[b] > 0)
            t, a, b, a1, b1 = t[go], a[go], b[go], a1[go], b1[go]
            if t.numel() == 0:
                break
            a = G.in_col[G.in_off[a] + _mulhi(a1, G.deg_in[a])]
            b = G.in_col[G.in_off[b] + _mulhi(b1, G.deg_in[b])]
            same = a == b
            met += int(same.sum())
            t, a, b = t[~same], a[~same], b[~same]
    return met
