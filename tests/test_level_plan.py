"""The level loop's column plan (csrc/level_plan.h, plain C++) against its rules written out plainly: heirs, chains
coloured first fit, push blocks grouped by parent, accumulate parts, zero masks.  Random trees, nodes exported in random
order; every number must be equal."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_06955_gb300", "csrc")
HARNESS = r"""
#include "level_plan.h"
#include <cstdio>
static void put(const char *name, const std::vector<int32_t> &v) {
    printf("%s", name);
    for (int32_t x : v) printf(" %d", x);
    printf("\n");
}
int main() {
    int N, B, D1, trees;
    long long cap;
    if (scanf("%d", &trees) != 1) return 1;
    ps::LevelPlan P;  // one object for all trees, as a workspace keeps it
    while (trees-- > 0) {
        if (scanf("%d %lld %d %d", &N, &cap, &B, &D1) != 4) return 1;
        std::vector<int32_t> e(N), p(N), t(N);
        for (int i = 0; i < N; ++i)
            if (scanf("%d %d %d", &e[i], &p[i], &t[i]) != 3) return 1;
        const bool ok = P.build(N, e.data(), p.data(), t.data(), cap, B, D1, [](int32_t r) {
            int32_t w = 1;
            while (w < r) w *= 2;
            return w;
        });
        printf("ok %d\n", (int)ok);
        if (!ok) continue;
        put("width", P.width), put("dw", P.dw), put("nfull", P.nfull), put("tail", P.tail), put("hinh", P.hinh);
        put("h0", P.h0), put("cols", P.cols), put("rho", P.rho), put("ent", P.ent), put("col", P.col);
        put("zmask", P.zmask), put("zoff", P.zoff), put("zany", P.zany);
        put("p1dst", P.p1dst), put("p1src", P.p1src), put("p2dst", P.p2dst), put("p2src", P.p2src);
        put("p1_at", P.p1_at), put("p2_at", P.p2_at);
        put("acc_src", std::vector<int32_t>(P.acc_src.begin(), P.acc_src.end()));
    }
}
"""


def tree(rng, B, walks, fan, keep, L):
    """Walk prefixes: {entry: (parent entry, depth, query, height)} with distinct random entries."""
    nodes, child = [[-1, 0, q, 0] for q in range(B)], {}
    for k in range(walks):
        x = k % B
        for _ in range(L):
            if nodes[x][1] > 0 and rng.random() > keep:
                break
            key = (x, int(rng.integers(fan)))
            if key not in child:
                child[key] = len(nodes)
                nodes.append([x, nodes[x][1] + 1, nodes[x][2], 0])
            x = child[key]
    for i in range(len(nodes) - 1, -1, -1):
        p = nodes[i][0]
        if p >= 0:
            nodes[p][3] = max(nodes[p][3], nodes[i][3] + 1)
    cap = 64
    while cap < 2 * len(nodes):
        cap *= 2
    at = rng.permutation(cap)[:len(nodes)]
    return {int(at[i]): (int(at[x[0]]) if x[0] >= 0 else -1, x[1], x[2], x[3]) for i, x in enumerate(nodes)}, cap


def plan(t, B, D1):
    dense = {e for e, (p, d, q, h) in t.items() if h >= 3 or (d == 0 and h >= 2)}
    own = sorted(dense | {e for e, (p, d, q, h) in t.items() if h == 2 and d > 0})
    dep = {e: t[e][1] for e in own}
    par = {e: t[e][0] for e in own}
    kids = {e: [] for e in own}
    for x in own:
        if par[x] >= 0:
            kids[par[x]].append(x)

    def depth_below(e):  # nodes on the longest path of dense descendants
        return max((1 + depth_below(x) for x in kids[e] if x in dense), default=0)
    chain = {e: depth_below(e) for e in dense}
    heir = {}
    for e in dense:
        dk, pk = [x for x in kids[e] if x in dense], [x for x in kids[e] if x not in dense]
        if dk:
            heir[e] = min(dk, key=lambda x: (-chain[x], x))
        elif pk:
            heir[e] = min(pk)
    inherits = set(heir.values())
    chains = []
    for e in dense - inherits:
        path = [e]
        while path[-1] in heir:
            path.append(heir[path[-1]])
        chains.append((dep[e] + len(path) - 1, dep[e], e, path))
    col, tops = {}, []
    for bottom, top, _, path in sorted(chains, key=lambda c: (-c[0], c[1], c[2])):
        c = next((i for i, x in enumerate(tops) if x > bottom + 1), len(tops))
        if c == len(tops):
            tops.append(top)
        tops[c] = min(tops[c], top)
        for x in path:
            col[x] = c
    o = {k: [] for k in ("width dw nfull tail hinh h0 cols zmask zoff zany p1dst p1src p2dst p2src p1_at p2_at "
                         "acc_src").split()}
    for d in range(D1):
        w = max((col[e] + 1 for e in dense if dep[e] == d), default=0)
        full, rem = (w // 32 + 1, 0) if w % 32 > 16 else (w // 32, w % 32)
        tail = 0 if rem == 0 else 1 << (rem - 1).bit_length()
        for k, v in (("width", w), ("nfull", full), ("tail", tail), ("dw", 32 * full + tail)):
            o[k].append(v)
    rho = [-1] * B
    for e in dense:
        if dep[e] == 0:
            rho[t[e][2]] = col[e]
    for d in range(D1):
        push = [e for e in own if e not in dense and dep[e] == d]
        o["hinh"].append(sum(e in inherits for e in push))
        o["h0"].append((max(1, o["dw"][d], o["dw"][d - 1] if d else 0) + 3) // 4 * 4)
        rest = sorted((e for e in push if e not in inherits), key=lambda e: (col[par[e]], e))
        for i, e in enumerate(rest):
            col[e] = o["h0"][d] + i
        o["cols"].append((o["h0"][d] + len(rest) + 3) // 4 * 4)
    zoff = 0
    for d in range(D1):
        o["p1_at"].append(len(o["p1dst"]))
        o["p2_at"].append(len(o["p2dst"]))
        o["acc_src"].append(0)
        for e in sorted((e for e in dense if dep[e] == d), key=lambda e: col[e]):
            src = sorted(col[x] for x in kids[e] if x not in inherits)
            if not src and e in heir:
                continue
            o["acc_src"][d] += len(src)
            parts = [src[i:i + 4] for i in range(0, len(src), 4)] or [[]]
            for i, part in enumerate(parts):
                k = "p1" if i == 0 else "p2"
                o[k + "dst"].append(col[e] | (1 << 30 if i == 0 and e not in heir else 0))
                o[k + "src"] += part + [-1] * (4 - len(part))
        words = [0] * ((o["dw"][d] + 31) // 32)
        for e in inherits - dense:
            if dep[e] == d and col[e] < o["dw"][d]:
                words[col[e] // 32] |= 1 << col[e] % 32
        o["zoff"].append(zoff)
        zoff += len(words)
        o["zany"].append(int(any(words)))
        o["zmask"] += [w - (1 << 32) if w >> 31 else w for w in words]
    o["p1_at"].append(len(o["p1dst"]))
    o["p2_at"].append(len(o["p2dst"]))
    o["zoff"].append(zoff)
    o.update(rho=rho, ent=own, col=[col[e] for e in own])
    return dense, o


def test_plan_follows_its_rules(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(HARNESS)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    rng = np.random.default_rng(7)
    shapes = [(1, 1, 1, 1.0, 5), (1, 40, 2, 0.8, 12), (2, 300, 4, 0.77, 20), (3, 900, 25, 0.9, 9), (1, 60, 1, 1.0, 30),
              (2, 7, 3, 0.0, 4), (1, 2500, 60, 0.8, 64), (4, 1500, 3, 0.95, 14)]
    want, text = [], ["%d" % len(shapes)]
    for B, walks, fan, keep, L in shapes:
        t, cap = tree(rng, B, walks, fan, keep, L)
        D1 = L + 2
        dense, o = plan(t, B, D1)
        want.append(o)
        text.append("%d %d %d %d" % (len(o["ent"]), cap, B, D1))
        for e in rng.permutation(np.array(o["ent"], np.int64)):
            p, d, q, _ = t[int(e)]
            text.append("%d %d %d" % (e, p if d > 0 else -1 - q, 2 * d + (int(e) in dense)))
    out = subprocess.run([str(exe)], input="\n".join(text), capture_output=True, text=True, check=True).stdout
    got, cur = [], None
    for line in out.splitlines():
        k, *v = line.split()
        if k == "ok":
            assert v == ["1"]
            cur = {}
            got.append(cur)
        else:
            cur[k] = [int(x) for x in v]
    assert len(got) == len(want) and max(len(o["ent"]) for o in want) > 500
    for o, g in zip(want, got):
        assert set(o) == set(g)
        for k in o:
            assert o[k] == g[k], k
