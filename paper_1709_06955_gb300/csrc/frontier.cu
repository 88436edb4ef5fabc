// Frontier PROBE engine: every walk prefix of a call's reverse-reachability trees probed on its own, as Alg. 4
// runs Alg. 2, with Pruning Rule 2 (Sec. 4.1) and the best-of-both switch of Sec. 4.4.
//
// A probe is a tree node r_q (q >= 2) of weight w, the prefix (u_1..u_q); it runs levels j = 0..q-2 of
// Alg. 2.  All probes of a call advance one level per round.  A probe's frontier H_j is a segment of entries (out-list,
// score, first work item); its work items are its (entry, out-edge) pairs.  A round:
//   check    Sec. 4.4 a level early (k_fr_check)
//   plan     Sec. 4.4: a probe whose out-degree sum exceeds c0 * w * n leaves the deterministic rounds (Alg. 3 then
//            runs on its whole partial walk once per walk through the tree node, rand_probe.cu); the others get a class
//   tasks    the class's task list, and room for the probe's next segment
//   expand   every entry x pushes sqrt(c)/|I(v)| * Score(x) to each v in O(x), v != u_{q-j-1}; Pruning Rule 2 is
//            applied to the sums as they are written (Rule 2 of level j + 1), and entries that are pruned or have no
//            out-edges are not written at all
// The classes, by the bound D = min(out-degree sum, n) on the next frontier:
//   last     the probe's last level: pushes go straight into its query's estimate with weight w, or, for one query on a
//            graph of a few slabs, through sums in shared memory (k_fr_last)
//   single   one entry: its targets are distinct, so they are written as they come
//   warp, block, mid, wide   a table in shared memory (up to kWarpD, kBlockD, kMidD, kPartD entries); a wide probe's
//            targets are split by hash into up to kMaxParts parts, each a block that scans all of the probe's items and
//            keeps its own
//   slab     a sum for every node in shared memory (no keys, no search) when D is at least a quarter of n; the nodes of
//            a larger graph are dealt to up to kSlabParts parts
//   global   larger: open addressing over a power of two of slots in device memory, or a dense slab of n slots when D
//            is a sizeable fraction of n, swept into the next segment by a second kernel, which empties it
// Why: a global table costs an item two random sectors, and its sweeps read every slot; with one table per level in
// device memory the expansion and its compaction were 90 % of this engine's time.  Scanning a probe's items again costs
// a coalesced read and a hash; at six parts the two cost the same (Thm. 2's split on 150,000 nodes, ms per query: 16.9 at
// 6 parts, 18.2 at 8, 51.7 at 16; at 4 parts 17.3).  What bounds it now: the
// tables' scans of items (issue slots), and for batches and large graphs the last level's 64-bit atomics on the estimates
// (5e10 a second).
// Measured, before and after (one table per level in device memory): one eps_a = 0.1 query with Rule 2, 150,000 nodes
// 24.4 -> 14.8 ms (k_fr_last: another query 16.5 -> 14.4), 10,000 nodes 21.7 -> 9.6 (without k_fr_last); 64 mixed-eps
// switch queries on R-MAT 2^22: expansion, compaction and scans 405 -> 18 ms (the early switch: 95 of the 123 ms left
// without it).
//
// Scores are FP32 products accumulated in 2^-44 fixed point (64-bit sums; in shared memory a 32-bit low half whose
// carries go to the high half).  The sums are exact whatever order the adds land in, so the frontier sets, the pruning
// and switch decisions and the estimates are the same alone and in any batch, and a run repeats bit for bit.  Every
// score is at most 1 and every query's estimate sum at most n_r, so values stay below 2^62 for n_r <= 2^18 (checked by
// the host).
#include <algorithm>

#include "internal.cuh"

namespace ps {

namespace {

constexpr int kThreads = 256;
constexpr int kSweepTile = 4096;   // global-table slots per block of the sweep
constexpr int kFrSteps = 4;        // steps of 32 items whose loads go out together
constexpr int kCheckItems = 512;   // work items the early switch looks at

__device__ __forceinline__ float fx_to_f(long long v) { return __ll2float_rn(v) * __int_as_float((127 - kFixShift) << 23); }
__device__ __forceinline__ long long f_to_fx(float x) { return __float2ll_rn(x * __int_as_float((127 + kFixShift) << 23)); }

__device__ __forceinline__ uint32_t node_hash(int32_t v) {
    return (uint32_t)(((unsigned long long)(uint32_t)v * 0x9E3779B97F4A7C15ull) >> 32);
}

// a bijection of 32 bits (xor-shifts and odd multiplies, the finaliser of A. Appleby's MurmurHash3): the shared tables
// take their slot from its low bits and the part from its high bits, and splitting a part always separates distinct
// nodes in the end
__device__ __forceinline__ uint32_t mix32(uint32_t h) {
    h ^= h >> 16;
    h *= 0x85EBCA6Bu;
    h ^= h >> 13;
    h *= 0xC2B2AE35u;
    return h ^ (h >> 16);
}

// Rule 2 keeps an entry of score val at level j of a probe of length q when val * sqrt(c)^(q-j-1) > eps_p
__device__ __forceinline__ bool rule2_keeps(float val, const float *pw, float eps_p, int32_t q, int32_t j) {
    return eps_p <= 0.f || val * pw[q - j - 1] > eps_p;
}

// H_0 = {(u_q, 1)} for every probe; the first excluded node is u_{q-1}, the parent's
__global__ void k_fr_init(TrieTable t, FrontierProbes P, const int64_t *__restrict__ out_off,
                          const float *__restrict__ pw, float eps_p, FrontierEntry *list) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= P.P) return;
    const int32_t s = P.slot[p], x = t.node[s];
    const uint32_t beg = (uint32_t)out_off[x];
    uint32_t deg = (uint32_t)out_off[x + 1] - beg;
    if (!rule2_keeps(1.f, pw, eps_p, t.depth[s], 0)) deg = 0;
    list[p] = FrontierEntry{beg, 0u, deg, 1.f};
    P.beg[p] = p;
    P.packed[p] = deg ? ((unsigned long long)deg << kFrCountBits) + 1ull : 0ull;
    P.anc[p] = t.parent[s];
    P.lev[p] = 0;
    P.state[p] = 0;
}

__device__ __forceinline__ unsigned long long warp_sum(unsigned long long x) {
    for (int o = 16; o; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
}

// Per probe of [p0, p1): the switch decision (Sec. 4.4), the class and its tasks, and the range's totals.
// thr[w] = floor(c0 * w * n) (host FP64); the probe switches when its out-degree sum exceeds thr[w].  Planning a range
// again (after a part of it was deferred) decides the same again.
__global__ void __launch_bounds__(kThreads) k_fr_plan(TrieTable t, FrontierProbes P, int32_t p0, int32_t p1,
                                                      int32_t j, int32_t n, const long long *__restrict__ thr,
                                                      uint8_t *t_sw, unsigned long long *totals) {
    const int32_t p = p0 + blockIdx.x * blockDim.x + threadIdx.x;
    unsigned long long pk = 0;
    if (p < p1) pk = P.packed[p];
    const unsigned long long d = pk >> kFrCountBits, cnt = pk & kFrCountMask;
    int32_t cls = kFrNone;
    unsigned long long nt = 0, D = 0, slots = 0, sweeps = 0;
    if (d > 0) {
        const int32_t s = P.slot[p];
        if (thr && (long long)d > thr[t.weight[s]]) {
            P.state[p] |= kProbeSwitched;
            t_sw[s] = 1;
        } else {
            int32_t a = P.anc[p];
            for (int32_t l = P.lev[p]; l < j; ++l) a = t.parent[a];  // the excluded ancestor moves up a level at a time
            P.anc[p] = a;
            P.lev[p] = j;
            P.ex[p] = t.node[a];  // level j excludes u_{q-j-1}
            const unsigned long long chunks = (d + kFrChunk - 1) / kFrChunk;
            D = d < (unsigned long long)n ? d : (unsigned long long)n;
            if (j == t.depth[s] - 2) {
                cls = kFrLast, nt = chunks, D = 0;
            } else if (cnt == 1) {
                cls = kFrSingle, nt = chunks;
            } else {
                unsigned long long r = 2;  // the table the probe's next frontier needs, wherever it lies
                while (r < 2 * D) r <<= 1;
                slots = r;
                if (D <= kWarpD) {
                    cls = kFrWarp, nt = 1;
                } else if (D <= kBlockD) {
                    cls = kFrBlock, nt = 1;
                } else if (4 * D >= (unsigned long long)n && n <= (int32_t)(kSlabN * kSlabParts)) {
                    cls = kFrSlab, nt = (n + kSlabN - 1) / kSlabN;
                } else if (D <= kMidD) {
                    cls = kFrMid, nt = 1;
                } else if (D <= (unsigned long long)kPartD * kMaxParts) {
                    cls = kFrWide, nt = (D + kPartD - 1) / kPartD;
                } else {
                    cls = kFrGlobal, nt = chunks;
                    if (4 * D >= (unsigned long long)n) {  // dense slab: slot v holds node v
                        P.state[p] |= kProbeDense;
                        slots = n;
                    } else {
                        P.state[p] &= ~kProbeDense;
                    }
                    P.rsize[p] = (long long)slots;
                    sweeps = (slots + kSweepTile - 1) / kSweepTile;
                }
            }
        }
    }
    if (p < p1) {
        P.cls[p] = cls;
        P.nt[p] = (uint32_t)nt;
    }
    const int lane = threadIdx.x & 31;
    for (int c = kFrNone + 1; c < kFrClasses; ++c) {
        if (c == kFrSweep) continue;
        if (!__any_sync(0xffffffffu, cls == c)) continue;
        const unsigned long long v = warp_sum(cls == c ? nt : 0ull);
        if (lane == 0) atomicAdd(totals + c, v);
    }
    const unsigned long long live = cls != kFrNone ? d : 0ull;
    const unsigned long long vs[6] = {sweeps, D, slots, cls == kFrGlobal ? slots : 0ull, live, cls == kFrLast ? d : 0ull};
    const int at[6] = {kFrSweep, kFrTotD, kFrTotSlots, kFrTotGlobal, kFrTotItems, kFrTotLast};
    for (int k = 0; k < 6; ++k) {
        const unsigned long long v = warp_sum(vs[k]);
        if (lane == 0 && v) atomicAdd(totals + at[k], v);
    }
    const unsigned long long ce = warp_sum(cls != kFrNone ? cnt : 0ull);
    if (lane == 0 && ce) atomicAdd(totals + kFrTotEntries, ce);
}

// exclusive place of v among the warp's lanes on a shared counter, with one atomic per warp
__device__ __forceinline__ unsigned long long warp_reserve(unsigned long long v, unsigned long long *counter) {
    const int lane = threadIdx.x & 31;
    unsigned long long incl = v;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    unsigned long long base = 0;
    if (lane == 31 && incl) base = atomicAdd(counter, incl);
    return __shfl_sync(0xffffffffu, base, 31) + incl - v;
}

// The task lists of the range's classes (class c's tasks from base[c]), room for every probe's next segment (D
// entries), and the global tables' regions.  cursor holds one counter per class and for the entries and slots, all 0.
__global__ void __launch_bounds__(kThreads) k_fr_tasks(FrontierProbes P, int32_t p0, int32_t p1, int32_t n,
                                                       FrontierBases base, unsigned long long *cursor,
                                                       FrontierTask *tasks) {
    const int32_t p = p0 + blockIdx.x * blockDim.x + threadIdx.x;
    int32_t cls = kFrNone;
    uint32_t nt = 0;
    unsigned long long D = 0;
    if (p < p1) {
        cls = P.cls[p];
        nt = P.nt[p];
        const unsigned long long d = P.packed[p] >> kFrCountBits;
        if (cls != kFrNone && cls != kFrLast) D = d < (unsigned long long)n ? d : (unsigned long long)n;
        P.packed_nx[p] = 0;
    }
    const unsigned long long at = warp_reserve(D, cursor + kFrTotD);
    if (p < p1) P.beg_nx[p] = (long long)at;
#pragma unroll
    for (int c = kFrNone + 1; c < kFrSweep; ++c) {
        if (!__any_sync(0xffffffffu, cls == c)) continue;
        const unsigned long long pos = warp_reserve(cls == c ? nt : 0u, cursor + c);
        if (cls == c)
            for (uint32_t k = 0; k < nt; ++k) tasks[base.at[c] + pos + k] = FrontierTask{p, k};
    }
    if (__any_sync(0xffffffffu, cls == kFrGlobal)) {
        const unsigned long long r = cls == kFrGlobal ? (unsigned long long)P.rsize[p] : 0ull;
        const unsigned long long off = warp_reserve(r, cursor + kFrTotGlobal);
        const uint32_t ns = (uint32_t)((r + kSweepTile - 1) / kSweepTile);
        const unsigned long long pos = warp_reserve(ns, cursor + kFrSweep);
        if (cls == kFrGlobal) {
            P.roff[p] = (long long)off;
            for (uint32_t k = 0; k < ns; ++k) tasks[base.at[kFrSweep] + pos + k] = FrontierTask{p, k};
        }
    }
}

// Runs f(want, v, aux(v), score) over the work items [t0, t1) of a segment of cnt entries and d items, 32 at a time, all
// lanes together; `want(v)` says whether the lane's target matters (aux(v) is loaded then, else 0).  The warp holds a
// window of 32 entries, one per lane.  A step's entry starts form a 32-bit mask (one warp reduction), whose set bits up
// to a lane count the entries to the lane's own, and two shuffles bring that entry's out-list and score; so kFrSteps
// steps' targets are loaded together, then their aux, and a warp waits for two gathers per 32 kFrSteps items.  (With a
// search and an entry load per 32 items it waited for three, and the tables' kernels ran a third as fast.)
template <class Want, class Aux, class F>
__device__ __forceinline__ void fr_items(const DeviceGraph &g, const FrontierEntry *__restrict__ seg, uint32_t cnt,
                                         uint32_t d, uint32_t t0, uint32_t t1, const Want &want, const Aux &aux,
                                         const F &f) {
    using A = decltype(aux(0));
    if (t0 >= t1) return;
    const int lane = threadIdx.x & 31;
    uint32_t e = 0;  // the entry of item t0: the last with first <= t0, by a 32-way search
    for (uint32_t span = cnt; span > 1;) {
        const uint32_t step = (span + 31) / 32;
        const unsigned le = __ballot_sync(0xffffffffu, lane * step < span && seg[e + lane * step].first <= t0);
        const uint32_t k = 31 - __clz(le);  // lane 0 always holds
        e += k * step;
        span = min(step, span - k * step);
    }
    for (uint32_t t = t0; t < t1; e += 32) {
        FrontierEntry en = FrontierEntry{0u, d, 0u, 0.f};  // past the last entry: starts at the end
        if (e + lane < cnt) en = seg[e + lane];
        const uint32_t base = en.out_beg - en.first;
        const uint32_t lim = min(t1, __shfl_sync(0xffffffffu, en.first + en.deg, 31));  // the window's items end here
        uint32_t before = __popc(__ballot_sync(0xffffffffu, en.first < t));  // entries of the window that start before t
        while (t < lim) {
            int32_t v[kFrSteps];
            float val[kFrSteps];
            bool on[kFrSteps];
            A x[kFrSteps];
#pragma unroll
            for (int u = 0; u < kFrSteps; ++u) {
                const uint32_t tt = t + 32 * u, off = en.first - tt;
                const unsigned starts = __reduce_or_sync(0xffffffffu, off < 32u && tt < lim ? 1u << off : 0u);
                const uint32_t r = before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1;
                const uint32_t col = __shfl_sync(0xffffffffu, base, r & 31);
                val[u] = __shfl_sync(0xffffffffu, en.val, r & 31);
                on[u] = tt + lane < lim;
                v[u] = on[u] ? __ldg(g.out_col + (uint32_t)(col + tt + lane)) : 0;
                before += __popc(starts);
            }
#pragma unroll
            for (int u = 0; u < kFrSteps; ++u) {
                on[u] = on[u] && want(v[u]);
                x[u] = on[u] ? aux(v[u]) : A(0);
            }
#pragma unroll
            for (int u = 0; u < kFrSteps; ++u) f(on[u], v[u], x[u], val[u]);
            t = min(lim, t + 32 * kFrSteps);
        }
    }
}

// Sec. 4.4 a level early: a probe whose next frontier is certain to exceed c0 * w * n switches now.  The switch reads
// the out-degree sum of the next frontier's distinct nodes, a sum that only grows, so the first few hundred work items
// decide most probes: on R-MAT graphs with c0 = 0.01 nine probes of ten that expand a level switch at the next, after
// an expansion of tens of thousands of items that nothing used.  A warp per probe, the nodes met so far in shared
// memory, up to kCheckItems items.  Only without Rule 2 (which could prune a node met here from the sum).
__global__ void __launch_bounds__(kThreads) k_fr_check(DeviceGraph g, TrieTable t, FrontierProbes P, int32_t p0,
                                                       int32_t p1, int32_t j, const FrontierEntry *src,
                                                       const long long *__restrict__ thr, uint8_t *t_sw) {
    __shared__ uint32_t s_keys[kThreads / 32][2 * kCheckItems];
    uint32_t *keys = s_keys[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int64_t wi = p0 + ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5);
    if (wi >= p1) return;
    const int32_t p = (int32_t)wi;
    const unsigned long long pk = P.packed[p];
    const uint32_t d = (uint32_t)(pk >> kFrCountBits), cnt = (uint32_t)(pk & kFrCountMask);
    if (d == 0) return;
    const int32_t s = P.slot[p];
    const long long limit = thr[t.weight[s]];
    if ((long long)d > limit || j >= t.depth[s] - 2) return;  // the plan decides this level; a last level has no next
    int32_t a = P.anc[p];
    for (int32_t l = P.lev[p]; l < j; ++l) a = t.parent[a];
    const int32_t ex = t.node[a];
    for (int i = lane; i < 2 * kCheckItems; i += 32) keys[i] = 0u;
    __syncwarp();
    const uint32_t end = min(d, (uint32_t)kCheckItems);
    unsigned long long sum = 0;
    for (uint32_t t0 = 0; t0 < end; t0 += 128) {
        fr_items(
            g, src + P.beg[p], cnt, d, t0, min(end, t0 + 128u), [&](int32_t v) { return v != ex; },
            [&](int32_t v) { return (uint32_t)(g.out_off[v + 1] - g.out_off[v]); },
            [&](bool on, int32_t v, uint32_t deg, float) {
                if (!on || deg == 0) return;
                const uint32_t key = (uint32_t)v + 1u;
                uint32_t h = mix32((uint32_t)v) & (2 * kCheckItems - 1);
                for (int probe = 0; probe < 2 * kCheckItems; ++probe) {  // at most half full
                    const uint32_t k = atomicCAS(keys + h, 0u, key);
                    if (k == 0u) sum += deg;
                    if (k == 0u || k == key) return;
                    h = (h + 1) & (2 * kCheckItems - 1);
                }
            });
        if ((long long)warp_sum(sum) > limit) {
            if (lane == 0) {
                P.state[p] |= kProbeSwitched;
                P.packed[p] = 0;
                t_sw[s] = 1;
            }
            return;
        }
    }
}

// Appends the lanes' entries (deg > 0) to a probe's next segment, in the packed counter's order; all lanes together
__device__ __forceinline__ void fr_append(uint32_t beg, uint32_t deg, float val, unsigned long long *packed,
                                          FrontierEntry *seg) {
    const unsigned m = __ballot_sync(0xffffffffu, deg > 0);
    if (!m) return;
    const int lane = threadIdx.x & 31;
    uint32_t incl = deg;
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    unsigned long long base = 0;
    if (lane == 31) base = atomicAdd(packed, ((unsigned long long)incl << kFrCountBits) + __popc(m));
    base = __shfl_sync(0xffffffffu, base, 31);
    if (deg > 0)
        seg[(base & kFrCountMask) + __popc(m & ((1u << lane) - 1u))] =
            FrontierEntry{beg, (uint32_t)(base >> kFrCountBits) + incl - deg, deg, val};
}

// last level and single-entry probes: a warp per chunk of kFrChunk items
template <bool LAST>
__global__ void __launch_bounds__(kThreads) k_fr_direct(DeviceGraph g, TrieTable t, FrontierProbes P, FrontierLevel a,
                                                        int64_t task0, int64_t ntasks) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= ntasks) return;
    const FrontierTask tk = a.tasks[task0 + i];
    const int32_t p = tk.p, s = P.slot[p], ex = P.ex[p];
    const unsigned long long pk = P.packed[p];
    const uint32_t d = (uint32_t)(pk >> kFrCountBits), cnt = (uint32_t)(pk & kFrCountMask);
    const FrontierEntry *seg = a.src + P.beg[p];
    const uint32_t t0 = tk.part * (uint32_t)kFrChunk, t1 = min(d, t0 + (uint32_t)kFrChunk);
    auto want = [&](int32_t v) { return v != ex; };
    auto weight = [&](int32_t v) { return __ldg(g.w + v); };
    if (LAST) {
        unsigned long long *acc = a.acc + (int64_t)t.query[s] * g.n;
        const long long w = t.weight[s];
        fr_items(g, seg, cnt, d, t0, t1, want, weight, [&](bool on, int32_t v, float wv, float val) {
            if (on) atomicAdd(acc + v, (unsigned long long)(f_to_fx(wv * val) * w));
        });
    } else {
        const int32_t q = t.depth[s];
        unsigned long long *packed = P.packed_nx + p;
        FrontierEntry *out = a.dst + P.beg_nx[p];
        fr_items(g, seg, cnt, d, t0, t1, want, weight, [&](bool on, int32_t v, float wv, float val) {
            const float sc = fx_to_f(f_to_fx(wv * val));
            uint32_t beg = 0, deg = 0;
            if (on && rule2_keeps(sc, a.pw, a.eps_p, q, a.j + 1)) {
                beg = (uint32_t)g.out_off[v];
                deg = (uint32_t)g.out_off[v + 1] - beg;
            }
            fr_append(beg, deg, sc, packed, out);
        });
    }
}

// The last level of one query's call on a graph of at most kLastParts slabs: the estimates' 64-bit adds in the L2 (5e10 a
// second) were the engine's largest part there, so a block sums a slab of the nodes (v = part mod parts) in shared memory
// over its share of the tasks and adds the slab to the estimates once.  Every part reads every item, so it pays while the
// parts are few and the items many (see launch_fr_level).
constexpr int kLastThreads = 1024;
__global__ void __launch_bounds__(kLastThreads) k_fr_last(DeviceGraph g, TrieTable t, FrontierProbes P, FrontierLevel a,
                                                          int64_t task0, int64_t ntasks, uint32_t parts) {
    extern __shared__ uint32_t smem[];
    uint32_t *lo = smem, *hi = smem + kSlabN;
    const uint32_t part = blockIdx.x % parts, size = ((uint32_t)g.n + parts - 1) / parts;
    for (uint32_t i = threadIdx.x; i < size; i += kLastThreads) lo[i] = 0u, hi[i] = 0u;
    __syncthreads();
    const uint32_t inv = parts > 1 ? (uint32_t)((0x100000000ull + parts - 1) / parts) : 0u;
    auto index = [&](uint32_t v) { return parts > 1 ? __umulhi(v, inv) : v; };  // v / parts, exact for v < 2^32 / parts
    const int64_t step = (int64_t)(gridDim.x / parts) * (kLastThreads / 32);
    for (int64_t i = (int64_t)(blockIdx.x / parts) * (kLastThreads / 32) + (threadIdx.x >> 5); i < ntasks; i += step) {
        const FrontierTask tk = a.tasks[task0 + i];
        const int32_t p = tk.p, ex = P.ex[p];
        const unsigned long long pk = P.packed[p];
        const uint32_t d = (uint32_t)(pk >> kFrCountBits), cnt = (uint32_t)(pk & kFrCountMask);
        const uint32_t t0 = tk.part * (uint32_t)kFrChunk, t1 = min(d, t0 + (uint32_t)kFrChunk);
        const long long w = t.weight[P.slot[p]];
        fr_items(
            g, a.src + P.beg[p], cnt, d, t0, t1,
            [&](int32_t v) { return v != ex && (uint32_t)v - index((uint32_t)v) * parts == part; },
            [&](int32_t v) { return __ldg(g.w + v); },
            [&](bool on, int32_t v, float wv, float val) {
                if (!on) return;
                const unsigned long long c = (unsigned long long)(f_to_fx(wv * val) * w);
                const uint32_t h = index((uint32_t)v), cl = (uint32_t)c, old = atomicAdd(lo + h, cl);
                const uint32_t ch = (uint32_t)(c >> 32) + (old + cl < old ? 1u : 0u);
                if (ch) atomicAdd(hi + h, ch);
            });
    }
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < size; i += kLastThreads) {
        const unsigned long long c = ((unsigned long long)hi[i] << 32) | lo[i];
        if (c) atomicAdd(a.acc + (int64_t)i * parts + part, c);  // a sum above 0 belongs to a node below n
    }
}

// A table in shared memory, T threads a task.  Hash table: CAP slots of (node + 1, low and high half of the sum).  A part
// that holds more nodes than the table (the hash spreads a probe's nodes evenly, so only a contrived graph gets there)
// is split in two, as often as it takes: pieces are ranges of the bijection's value, so a range of CAP values always
// fits.  Slab: a sum for every node of the part (the nodes v = part mod parts), no keys and no search; a node whose
// every push rounded to 0 is marked in a bitmap, so membership stays exact.
template <int T, int CAP, bool SLAB>
__global__ void __launch_bounds__(T) k_fr_table(DeviceGraph g, TrieTable t, FrontierProbes P, FrontierLevel a,
                                                int64_t task0) {
    extern __shared__ uint32_t smem[];
    uint32_t *lo = smem, *hi = smem + CAP, *keys = smem + 2 * CAP;  // SLAB: keys is the bitmap
    __shared__ unsigned long long s_run;
    __shared__ unsigned long long s_red[T / 32];
    __shared__ int s_over;
    const FrontierTask tk = a.tasks[task0 + blockIdx.x];
    const int32_t p = tk.p, s = P.slot[p], ex = P.ex[p], q = t.depth[s];
    const unsigned long long pk = P.packed[p];
    const uint32_t d = (uint32_t)(pk >> kFrCountBits), cnt = (uint32_t)(pk & kFrCountMask);
    const FrontierEntry *seg = a.src + P.beg[p];
    FrontierEntry *out = a.dst + P.beg_nx[p];
    unsigned long long *packed = P.packed_nx + p;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    constexpr int NW = T / 32;
    const uint32_t per = ((d + NW - 1) / NW + 31) / 32 * 32;
    const uint32_t t0 = min(d, warp * per), t1 = min(d, t0 + per);
    const uint32_t parts = P.nt[p];
    // SLAB: v / parts by a multiplication, exact for v < 2^32 / parts
    const uint32_t inv = parts > 1 ? (uint32_t)((0x100000000ull + parts - 1) / parts) : 0u;
    auto index = [&](uint32_t v) { return parts > 1 ? __umulhi(v, inv) : v; };
    auto weight = [&](int32_t v) { return __ldg(g.w + v); };
    auto add = [&](uint32_t h, unsigned long long c) {  // the low half's carry goes to the high half
        const uint32_t cl = (uint32_t)c, old = atomicAdd(lo + h, cl);
        const uint32_t ch = (uint32_t)(c >> 32) + (old + cl < old ? 1u : 0u);
        if (ch) atomicAdd(hi + h, ch);
    };
    uint32_t size = CAP;
    if (SLAB) {
        size = ((uint32_t)g.n + parts - 1) / parts;
        size = (size + 31) / 32 * 32;
    } else if (parts == 1) {  // at most min(d, n) nodes: a smaller table when that is at most half its slots
        const uint32_t D = min(d, (uint32_t)g.n);
        while (size > 64 && size / 2 >= 2 * D) size >>= 1;
    }
    int lgs = 0;  // the part is taken in 2^lgs pieces
    for (uint32_t sub = 0; sub < (1u << lgs);) {
        for (uint32_t i = threadIdx.x; i < size; i += T) {
            lo[i] = 0u, hi[i] = 0u;
            if (!SLAB) keys[i] = 0u;
            else if (i < size / 32) keys[i] = 0u;
        }
        if (threadIdx.x == 0) s_over = 0, s_run = 0;
        __syncthreads();
        if (SLAB) {
            fr_items(
                g, seg, cnt, d, t0, t1,
                [&](int32_t v) { return v != ex && (uint32_t)v - index((uint32_t)v) * parts == tk.part; }, weight,
                [&](bool on, int32_t v, float wv, float val) {
                    if (!on) return;
                    const unsigned long long c = (unsigned long long)f_to_fx(wv * val);
                    const uint32_t h = index((uint32_t)v);
                    if (c) add(h, c);
                    else atomicOr(keys + (h >> 5), 1u << (h & 31));
                });
        } else {
            const uint32_t total = parts << lgs, target = (tk.part << lgs) + sub;
            fr_items(
                g, seg, cnt, d, t0, t1,
                [&](int32_t v) { return v != ex && (total == 1 || __umulhi(mix32((uint32_t)v), total) == target); },
                weight,
                [&](bool on, int32_t v, float wv, float val) {
                    if (!on) return;
                    const unsigned long long c = (unsigned long long)f_to_fx(wv * val);
                    const uint32_t key = (uint32_t)v + 1u;
                    uint32_t h = mix32((uint32_t)v) & (size - 1);
                    for (uint32_t probe = 0; probe < size; ++probe) {
                        uint32_t k = *reinterpret_cast<volatile uint32_t *>(keys + h);
                        if (k == 0u) {
                            k = atomicCAS(keys + h, 0u, key);
                            if (k == 0u) k = key;
                        }
                        if (k == key) {
                            add(h, c);
                            return;
                        }
                        h = (h + 1) & (size - 1);
                    }
                    s_over = 1;  // the part is larger than the table
                });
        }
        __syncthreads();
        if (!SLAB && s_over) {
            __syncthreads();
            ++lgs;
            sub <<= 1;
            continue;
        }
        // scores, Rule 2 and out-lists of the nodes found; then their places
        unsigned long long sum = 0;
        for (uint32_t i0 = threadIdx.x; i0 < size; i0 += 4 * T) {
            uint32_t node[4], beg[4], deg[4];
            float sc[4];
            bool hit[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * T;
                hit[u] = false;
                beg[u] = deg[u] = 0;
                if (i >= size) continue;
                if (SLAB) {
                    hit[u] = (lo[i] | hi[i]) != 0u || ((keys[i >> 5] >> (i & 31)) & 1u);
                    node[u] = i * parts + tk.part;
                } else {
                    hit[u] = keys[i] != 0u;
                    node[u] = keys[i] - 1u;
                }
                if (!hit[u]) continue;
                sc[u] = fx_to_f((long long)(((unsigned long long)hi[i] << 32) | lo[i]));
                if (!rule2_keeps(sc[u], a.pw, a.eps_p, q, a.j + 1)) continue;
                beg[u] = (uint32_t)g.out_off[node[u]];
                deg[u] = (uint32_t)g.out_off[node[u] + 1u];
            }
#pragma unroll
            for (int u = 0; u < 4; ++u) {
                const uint32_t i = i0 + u * T;
                if (!hit[u]) continue;
                deg[u] -= beg[u];
                if (!SLAB) keys[i] = beg[u];
                lo[i] = __float_as_uint(sc[u]);
                hi[i] = deg[u];
                if (deg[u]) sum += ((unsigned long long)deg[u] << kFrCountBits) + 1ull;
            }
        }
        sum = warp_sum(sum);
        if (lane == 0) s_red[warp] = sum;
        __syncthreads();
        if (threadIdx.x == 0) {
            unsigned long long tot = 0;
            for (int w = 0; w < NW; ++w) tot += s_red[w];
            s_run = tot ? atomicAdd(packed, tot) : 0ull;
        }
        __syncthreads();
        for (uint32_t i0 = warp * 32; i0 < size; i0 += T) {
            const uint32_t i = i0 + lane, deg = hi[i];
            uint32_t beg = 0;
            if (deg) beg = SLAB ? (uint32_t)g.out_off[i * parts + tk.part] : keys[i];
            fr_append(beg, deg, __uint_as_float(lo[i]), &s_run, out);
        }
        __syncthreads();
        ++sub;
    }
}

// global tables: a warp per chunk of items
__global__ void __launch_bounds__(kThreads) k_fr_global(DeviceGraph g, FrontierProbes P, FrontierLevel a, int64_t task0,
                                                        int64_t ntasks) {
    const int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    if (i >= ntasks) return;
    const FrontierTask tk = a.tasks[task0 + i];
    const int32_t p = tk.p, ex = P.ex[p];
    const unsigned long long pk = P.packed[p];
    const uint32_t d = (uint32_t)(pk >> kFrCountBits), cnt = (uint32_t)(pk & kFrCountMask);
    FrontierSlot *tab = a.tab + P.roff[p];
    const long long R = P.rsize[p];
    const bool dense = P.state[p] & kProbeDense;
    const uint32_t t0 = tk.part * (uint32_t)kFrChunk, t1 = min(d, t0 + (uint32_t)kFrChunk);
    fr_items(
        g, a.src + P.beg[p], cnt, d, t0, t1, [&](int32_t v) { return v != ex; },
        [&](int32_t v) { return __ldg(g.w + v); },
        [&](bool on, int32_t v, float wv, float val) {
            if (!on) return;
            const unsigned long long c = (unsigned long long)f_to_fx(wv * val);
            const int32_t key = v + 1;
            if (dense) {
                tab[v].key = key;
                atomicAdd(&tab[v].val, c);
                return;
            }
            long long h = node_hash(v) & (R - 1);
            for (long long probe = 0; probe < R; ++probe) {
                FrontierSlot &slot = tab[h];
                int32_t k = slot.key;
                if (k == 0) {
                    k = atomicCAS(&slot.key, 0, key);
                    if (k == 0) k = key;
                }
                if (k == key) {
                    atomicAdd(&slot.val, c);
                    break;
                }
                h = (h + 1) & (R - 1);
            }
        });
}

// the occupied slots of a tile of a region become entries of the probe's next segment, and the tile is emptied, so the
// table needs no clearing between passes
__global__ void __launch_bounds__(kThreads) k_fr_sweep(DeviceGraph g, TrieTable t, FrontierProbes P, FrontierLevel a,
                                                       int64_t task0) {
    const FrontierTask tk = a.tasks[task0 + blockIdx.x];
    const int32_t p = tk.p, q = t.depth[P.slot[p]];
    FrontierSlot *tab = a.tab + P.roff[p];
    const long long R = P.rsize[p], b0 = (long long)tk.part * kSweepTile;
    FrontierEntry *out = a.dst + P.beg_nx[p];
    unsigned long long *packed = P.packed_nx + p;
    for (int r = 0; r < kSweepTile; r += kThreads) {
        const long long k = b0 + r + threadIdx.x;
        uint32_t beg = 0, deg = 0;
        float sc = 0.f;
        if (k < R && tab[k].key != 0) {
            const int32_t v = tab[k].key - 1;
            sc = fx_to_f((long long)tab[k].val);
            if (rule2_keeps(sc, a.pw, a.eps_p, q, a.j + 1)) {
                beg = (uint32_t)g.out_off[v];
                deg = (uint32_t)g.out_off[v + 1] - beg;
            }
            *reinterpret_cast<ulonglong2 *>(tab + k) = make_ulonglong2(0ull, 0ull);
        }
        fr_append(beg, deg, sc, packed, out);
    }
}

// copies the segments of the probes [p0, p1) to the deferral stack, from entry *top on (a block per probe)
__global__ void __launch_bounds__(128) k_fr_defer(FrontierProbes P, int32_t p0, const FrontierEntry *src,
                                                  FrontierEntry *stack, unsigned long long *top) {
    __shared__ unsigned long long s_at;
    const int32_t p = p0 + blockIdx.x;
    const unsigned long long cnt = P.packed[p] & kFrCountMask;
    if (cnt == 0 || P.cls[p] == kFrNone) return;
    const long long from = P.beg[p];
    if (threadIdx.x == 0) s_at = atomicAdd(top, cnt);
    __syncthreads();
    for (unsigned long long k = threadIdx.x; k < cnt; k += blockDim.x) stack[s_at + k] = src[from + k];
    __syncthreads();
    if (threadIdx.x == 0) P.beg[p] = (long long)s_at;
}

__global__ void k_fr_count_switched(FrontierProbes P, unsigned long long *count) {
    const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
    const bool sw = p < P.P && (P.state[p] & kProbeSwitched);
    const unsigned m = __ballot_sync(0xffffffffu, sw);
    if ((threadIdx.x & 31) == 0 && m) atomicAdd(count, (unsigned long long)__popc(m));
}

// s(u, v) = (fixed-point deterministic sum + randomized member count) / n_r + shift, s(u, u) = 1
__global__ void k_fr_finalize(int32_t n, const int32_t *__restrict__ qnode, const unsigned long long *__restrict__ acc,
                              const int32_t *__restrict__ counts, const float *__restrict__ inv_nr,
                              const int32_t *__restrict__ ext2int, float shift, float *__restrict__ out) {
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t b = blockIdx.y;
    if (v >= n) return;
    const int64_t i = (int64_t)b * n + ext2int[v];
    long long tot = (long long)acc[i];
    if (counts) tot += (long long)counts[i] << kFixShift;
    float s = fx_to_f(tot) * inv_nr[b] + shift;
    if ((int32_t)v == qnode[b]) s = 1.f;
    out[(int64_t)b * n + v] = s;
}

inline unsigned blocks_for(int64_t count, int threads = kThreads) {
    return (unsigned)std::max<int64_t>(1, (count + threads - 1) / threads);
}

template <int T, int CAP, bool SLAB>
cudaError_t launch_table(const DeviceGraph &g, const TrieTable &t, const FrontierProbes &P, const FrontierLevel &a,
                         int64_t task0, int64_t ntasks, cudaStream_t s) {
    if (ntasks <= 0) return cudaSuccess;
    constexpr size_t bytes = SLAB ? (size_t)CAP * 8 + CAP / 8 : (size_t)CAP * 12;
    if (bytes > 48 * 1024) {
        const cudaError_t e =
            cudaFuncSetAttribute(k_fr_table<T, CAP, SLAB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
    }
    k_fr_table<T, CAP, SLAB><<<(unsigned)ntasks, T, bytes, s>>>(g, t, P, a, task0);
    return cudaSuccess;
}

}  // namespace

void launch_fr_init(TrieTable t, FrontierProbes P, const int64_t *out_off, const float *pw, float eps_p,
                    FrontierEntry *list, cudaStream_t s) {
    if (P.P > 0) k_fr_init<<<blocks_for(P.P), kThreads, 0, s>>>(t, P, out_off, pw, eps_p, list);
}
void launch_fr_check(const DeviceGraph &g, TrieTable t, FrontierProbes P, int32_t p0, int32_t p1, int32_t j,
                     const FrontierEntry *src, const long long *thr, uint8_t *t_sw, cudaStream_t s) {
    if (p1 > p0) k_fr_check<<<blocks_for(32 * (int64_t)(p1 - p0)), kThreads, 0, s>>>(g, t, P, p0, p1, j, src, thr, t_sw);
}
void launch_fr_plan(TrieTable t, FrontierProbes P, int32_t p0, int32_t p1, int32_t j, int32_t n,
                    const long long *thr, uint8_t *t_sw, unsigned long long *totals, cudaStream_t s) {
    if (p1 > p0) k_fr_plan<<<blocks_for(p1 - p0), kThreads, 0, s>>>(t, P, p0, p1, j, n, thr, t_sw, totals);
}
void launch_fr_tasks(FrontierProbes P, int32_t p0, int32_t p1, int32_t n, const FrontierBases &base,
                     unsigned long long *cursor, FrontierTask *tasks, cudaStream_t s) {
    if (p1 > p0) k_fr_tasks<<<blocks_for(p1 - p0), kThreads, 0, s>>>(P, p0, p1, n, base, cursor, tasks);
}
cudaError_t launch_fr_level(const DeviceGraph &g, TrieTable t, FrontierProbes P, const FrontierLevel &a,
                            const FrontierBases &base, const unsigned long long *ntasks, cudaStream_t s,
                            int64_t *launches) {
    auto n = [&](int c) { return (int64_t)ntasks[c]; };
    for (int c = kFrNone + 1; c < kFrClasses; ++c) *launches += n(c) > 0;
    if (n(kFrGlobal) > 0)
        k_fr_global<<<blocks_for(32 * n(kFrGlobal)), kThreads, 0, s>>>(g, P, a, base.at[kFrGlobal], n(kFrGlobal));
    static_assert(kPartD <= 16384 * 3 / 4 && kMidD <= 8192 * 3 / 4 && kBlockD <= 2048 * 3 / 4 && kWarpD <= 256 / 2,
                  "every class's next frontier fits its table");
    cudaError_t e = launch_table<1024, kSlabN, true>(g, t, P, a, base.at[kFrSlab], n(kFrSlab), s);
    if (e == cudaSuccess) e = launch_table<1024, 16384, false>(g, t, P, a, base.at[kFrWide], n(kFrWide), s);
    if (e == cudaSuccess) e = launch_table<512, 8192, false>(g, t, P, a, base.at[kFrMid], n(kFrMid), s);
    if (e == cudaSuccess) e = launch_table<128, 2048, false>(g, t, P, a, base.at[kFrBlock], n(kFrBlock), s);
    if (e == cudaSuccess) e = launch_table<32, 256, false>(g, t, P, a, base.at[kFrWarp], n(kFrWarp), s);
    if (e != cudaSuccess) return e;
    if (n(kFrSingle) > 0)
        k_fr_direct<false><<<blocks_for(32 * n(kFrSingle)), kThreads, 0, s>>>(g, t, P, a, base.at[kFrSingle],
                                                                              n(kFrSingle));
    // k_fr_last against k_fr_direct<true>, ms per query with Thm. 2's split of 0.1, 16 edges a node: 20,000 nodes (1 part)
    // 3.6 against 9.0, 60,000 (3) 8.6 / 14.5, 100,000 (5) 11.9 / 15.4, 150,000 (7) 13.6 / 15.1, 200,000 (9) 20.4 / 22.0,
    // 240,000 (10) 23.0 / 24.0.  Adding the slabs costs about as much as 4 million items' adds; tasks of few items cost
    // their start once per part.
    const uint32_t parts = ((uint32_t)g.n + kSlabN - 1) / kSlabN;
    if (n(kFrLast) > 0 && a.one_query && parts <= kLastParts && ntasks[kFrTotLast] >= kLastItems &&
        ntasks[kFrTotLast] >= kLastPerTask * ntasks[kFrLast]) {
        constexpr int bytes = (int)kSlabN * 8;
        e = cudaFuncSetAttribute(k_fr_last, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
        k_fr_last<<<parts * std::max(1u, 152u / parts), kLastThreads, bytes, s>>>(g, t, P, a, base.at[kFrLast],
                                                                                  n(kFrLast), parts);
    } else if (n(kFrLast) > 0)
        k_fr_direct<true><<<blocks_for(32 * n(kFrLast)), kThreads, 0, s>>>(g, t, P, a, base.at[kFrLast], n(kFrLast));
    if (n(kFrSweep) > 0) k_fr_sweep<<<(unsigned)n(kFrSweep), kThreads, 0, s>>>(g, t, P, a, base.at[kFrSweep]);
    return cudaSuccess;
}
void launch_fr_defer(FrontierProbes P, int32_t p0, int32_t p1, const FrontierEntry *src, FrontierEntry *stack,
                     unsigned long long *top, cudaStream_t s) {
    if (p1 > p0) k_fr_defer<<<(unsigned)(p1 - p0), 128, 0, s>>>(P, p0, src, stack, top);
}
void launch_fr_count_switched(FrontierProbes P, unsigned long long *count, cudaStream_t s) {
    cudaMemsetAsync(count, 0, sizeof(unsigned long long), s);
    if (P.P > 0) k_fr_count_switched<<<blocks_for(P.P), kThreads, 0, s>>>(P, count);
}
void launch_fr_finalize(int32_t n, int32_t B, const int32_t *qnode, const unsigned long long *acc, const int32_t *counts,
                        const float *inv_nr, const int32_t *ext2int, float shift, float *out, cudaStream_t s) {
    dim3 grid(blocks_for(n), (unsigned)B);
    k_fr_finalize<<<grid, kThreads, 0, s>>>(n, qnode, acc, counts, inv_nr, ext2int, shift, out);
}

}  // namespace ps
