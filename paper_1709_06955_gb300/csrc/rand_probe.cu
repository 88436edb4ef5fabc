// Randomized PROBE (Alg. 3) for every probe instance of a launch: instance (walk k, prefix length i) runs
// levels j = 0..i-2 over a frontier H_j of nodes (all with score 1).  At level j each candidate x != u_{i-j-1}
// samples one in-edge (v, x) of I(x) and joins H_{j+1} with probability sqrt(c) when v is in H_j
// (Alg. 3 lines 8-11); the draws use Philox counter (k, 2^24 | i << 8 | j, x, 0) with x the caller's node id,
// so the outcome of a candidate does not depend on how often or in which order it is evaluated.
//
// Candidates: Alg. 3 takes U = union of O(y), y in H_j, or V when that union is large (lines 4-7).  A node
// outside the union has no in-neighbour in H_j and can never be selected, so both choices give the same
// H_{j+1}; the kernels always evaluate the union, one work item per (frontier entry y, out-edge y -> x).
//
// x joins H_{j+1} when its sampled in-neighbour v lies in H_j.  Then the item (v, x) is itself among the level's work
// items, and it is the only item of x whose entry equals the sample.  So an item tests v == y and nothing else: every
// member is found by exactly one item, no set of H_j is looked up and no set of H_{j+1} is needed to drop repeats
// (hash sets for both took 60-80 % of this engine's time in random sectors and clears; see k_rand_level).
// The members of H_{i-1} are counted per query node; the estimate is count / n_r (Alg. 1 with randomized PROBE),
// exact in integers.
#include "internal.cuh"

namespace ps {

// ------------------------------------------------------------------------------------------------
// exclusive scan of int64 values (three passes: block sums, scan of the block sums, block scans)
// ------------------------------------------------------------------------------------------------
constexpr int kScanBlock = 1024;
constexpr int kScanItems = 4;  // per thread
constexpr int kScanTile = kScanBlock * kScanItems;

__device__ __forceinline__ long long block_exclusive_scan(long long v, long long *s_warp, long long *total) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    long long x = v;
    for (int o = 1; o < 32; o <<= 1) {
        const long long y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    if (warp == 0) {
        long long t = lane < (int)(blockDim.x >> 5) ? s_warp[lane] : 0;
        for (int o = 1; o < 32; o <<= 1) {
            const long long y = __shfl_up_sync(0xffffffffu, t, o);
            if (lane >= o) t += y;
        }
        s_warp[lane] = t;  // inclusive per warp
    }
    __syncthreads();
    const long long base = warp > 0 ? s_warp[warp - 1] : 0;
    *total = s_warp[(blockDim.x >> 5) - 1];
    __syncthreads();
    return base + x - v;
}

__global__ void __launch_bounds__(kScanBlock) k_scan_partials(const long long *__restrict__ in, int64_t count,
                                                              long long *__restrict__ partial) {
    __shared__ long long s_warp[32];
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    long long local = 0;
    for (int r = 0; r < kScanItems; ++r) {
        const int64_t i = base + (int64_t)r * kScanBlock + threadIdx.x;
        if (i < count) local += in[i];
    }
    long long total;
    block_exclusive_scan(local, s_warp, &total);
    if (threadIdx.x == 0) partial[blockIdx.x] = total;
}

// one block scans the block sums in place (any count, in chunks of kScanBlock)
__global__ void __launch_bounds__(kScanBlock) k_scan_partials_scan(long long *partial, int64_t nblocks) {
    __shared__ long long s_warp[32];
    __shared__ long long s_carry;
    if (threadIdx.x == 0) s_carry = 0;
    __syncthreads();
    for (int64_t c0 = 0; c0 < nblocks; c0 += kScanBlock) {
        const int64_t i = c0 + threadIdx.x;
        const long long v = i < nblocks ? partial[i] : 0;
        long long total;
        const long long ex = block_exclusive_scan(v, s_warp, &total);
        if (i < nblocks) partial[i] = s_carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) s_carry += total;
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kScanBlock) k_scan_final(const long long *__restrict__ in, int64_t count,
                                                           const long long *__restrict__ partial,
                                                           long long *__restrict__ out) {
    __shared__ long long s_warp[32];
    __shared__ long long s_carry;
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    if (threadIdx.x == 0) s_carry = partial[blockIdx.x];
    __syncthreads();
    for (int r = 0; r < kScanItems; ++r) {
        const int64_t i = base + (int64_t)r * kScanBlock + threadIdx.x;
        const long long v = i < count ? in[i] : 0;
        long long total;
        const long long ex = block_exclusive_scan(v, s_warp, &total);
        if (i < count) out[i] = s_carry + ex;
        __syncthreads();
        if (threadIdx.x == 0) s_carry += total;
        __syncthreads();
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) out[count] = s_carry;
}

int64_t scan64_partials_needed(int64_t count) { return (count + kScanTile - 1) / kScanTile + 1; }

// out[0..count] = exclusive prefix sums of in[0..count), out[count] = total.  partial holds
// scan64_partials_needed(count) entries.
void launch_scan64(const long long *in, int64_t count, long long *partial, long long *out, cudaStream_t s) {
    if (count <= 0) {
        cudaMemsetAsync(out, 0, sizeof(long long), s);
        return;
    }
    const int64_t nb = (count + kScanTile - 1) / kScanTile;
    k_scan_partials<<<(unsigned)nb, kScanBlock, 0, s>>>(in, count, partial);
    k_scan_partials_scan<<<1, kScanBlock, 0, s>>>(partial, nb);
    k_scan_final<<<(unsigned)nb, kScanBlock, 0, s>>>(in, count, partial, out);
}

// ------------------------------------------------------------------------------------------------
// probe instances
// ------------------------------------------------------------------------------------------------
__device__ __forceinline__ int32_t walk_query(const int32_t *walk_base, int32_t B, int32_t wid) {
    int32_t lo = 0, hi = B;
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (walk_base[mid] <= wid) lo = mid; else hi = mid;
    }
    return lo;
}

// Reserves a place in a level's list, and `deg` work items, for every lane with deg > 0.  The counter packs the entry
// count (low kRandCountBits) and the sum of the out-degrees, so one atomic per warp gives the entries their places and
// their first work items in the same order: the list comes with its prefix sums, and no scan runs.  `check` sums the
// degrees alone; the host compares the two to see an overflow of a packed field.  All 32 lanes call it together;
// returns the lane's place and sets its first item.
__device__ __forceinline__ long long rand_reserve(uint32_t deg, unsigned long long *packed, unsigned long long *check,
                                                  long long *item) {
    const unsigned mask = __ballot_sync(0xffffffffu, deg > 0);
    if (!mask) return 0;
    const int lane = threadIdx.x & 31;
    unsigned long long incl = deg;
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned long long y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    unsigned long long base = 0;
    if (lane == 31) {
        base = atomicAdd(packed, (incl << kRandCountBits) + (unsigned long long)__popc(mask));
        atomicAdd(check, incl);
    }
    base = __shfl_sync(0xffffffffu, base, 31);
    *item = (long long)((base >> kRandCountBits) + incl - deg);
    return (long long)(base & kRandCountMask) + __popc(mask & ((1u << lane) - 1u));
}

// instance (w, i) runs unless a filter is given and the tree slot of its prefix is not flagged
__device__ __forceinline__ bool inst_on(const int32_t *walk_slot, const uint8_t *t_sw, int32_t l_max, int32_t w, int32_t i) {
    return !walk_slot || t_sw[walk_slot[(int64_t)w * l_max + i - 1]];
}

__global__ void k_add_i32(int32_t *__restrict__ a, const int32_t *__restrict__ b, int64_t count) {
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count; i += (int64_t)gridDim.x * blockDim.x)
        a[i] += b[i];
}

// Instances (walk w, prefix length i), i = 2..len, and their level-0 entries {u_i}: one thread per (walk, i), so a
// long walk holds up no warp.  u_i is an in-neighbour of u_{i-1}, so its out-list is never empty.
__global__ void __launch_bounds__(256) k_inst_init(QueryBatch q, DeviceGraph g, const int32_t *__restrict__ lens,
                                                   int32_t w0, int32_t nw, int32_t l_max, int32_t max_len,
                                                   const int32_t *__restrict__ walks, RandList out,
                                                   unsigned long long *packed, unsigned long long *check,
                                                   const int32_t *__restrict__ walk_slot,
                                                   const uint8_t *__restrict__ t_sw) {
    const int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t span = max_len - 1;
    const int64_t wi = id / span;
    const int32_t w = w0 + (int32_t)wi, i = 2 + (int32_t)(id - wi * span);
    uint32_t deg = 0;
    RandEntry e = {};
    if (wi < nw && i <= lens[w] && inst_on(walk_slot, t_sw, l_max, w, i)) {
        e.y = walks[(int64_t)w * l_max + i - 1];   // H_0 = {u_i}
        e.ex = walks[(int64_t)w * l_max + i - 2];  // level 0 excludes u_{i-1}
        e.out_beg = (uint32_t)g.out_off[e.y];
        deg = (uint32_t)g.out_off[e.y + 1] - e.out_beg;
        e.id8 = (uint32_t)g.int2ext[e.y] >> g.rec_shift;
        e.len = i;
        e.walk = w;
        e.q = walk_query(q.walk_base, q.B, w);
        e.k = (uint32_t)(q.walk_k0[e.q] + (w - q.walk_base[e.q]));
    }
    long long item;
    const long long pos = rand_reserve(deg, packed, check, &item);
    if (deg > 0 && pos < out.cap) {
        out.ent[pos] = e;
        out.first[pos] = item;
    }
}

constexpr int kLevelThreads = 256;
constexpr int kLevelBuffer = 128;     // members a warp holds back before it appends them
constexpr int kLevelMaxItems = 4096;  // work items a warp takes at a time, at most

// One level.  A warp takes a run of consecutive work items (32 to kLevelMaxItems, so that a short level still spreads
// over the chip).  It holds the first items of the next 32 entries in registers; every entry has at least one item, so
// the entries of 32 items lie in that window and a lane finds its own by five shuffles.  Where one entry holds the next
// 64 items or more (the rule at level 0, whose entries are hubs), its items run through a pipeline of four stages --
// out-edge, record, draw, in-edge -- with a load of each in flight; else 32 items of several entries go at once.
// What bounds it: dependent random sectors (a record per item; an in-list entry for a fifth of them) at 32 warps per
// SM, then the ten Philox rounds (a third of the time at level 0 goes when they are left out).
// A top-k call of four queries at eps = 0.1 on R-MAT 2^20: 6.2 ms with hash sets (4.5 ms of level kernels, 0.55 ms of
// clears, two synchronisations a level); 3.0 without them; 2.3 with the records, the pipeline, self-contained entries
// (a level of 60 million items in 0.49 ms; 0.81 before) and appends gathered per warp.  64 mixed-eps queries with the
// switch on R-MAT 2^22: 332 ms of level kernels with hash sets, 115 now.
__global__ void __launch_bounds__(kLevelThreads, 4) k_rand_level(DeviceGraph g, const int32_t *__restrict__ walks,
                                                              int32_t l_max,
                                                              const uint32_t *__restrict__ qkey, uint32_t seed,
                                                              uint32_t t_keep, RandLevel L) {
    const unsigned long long packed_in = *L.packed_in;
    const long long F = (long long)(packed_in & kRandCountMask), E = (long long)(packed_in >> kRandCountBits);
    if (F == 0 || F > L.cur.cap || E > L.max_items) return;  // the host grows the list, or runs the range again
    const int lane = threadIdx.x & 31;
    const long long warp = (blockIdx.x * (long long)blockDim.x + threadIdx.x) >> 5;
    const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
    long long run = (E / nwarps + 31) / 32 * 32;
    run = run < 32 ? 32 : (run > kLevelMaxItems ? kLevelMaxItems : run);
    // A warp gathers its members in shared memory, as (its entry's number, node), and appends up to kLevelBuffer of
    // them with one atomic: an atomic per 32 items on the level's one counter, with the member's gathers behind it,
    // took a tenth of the call (2.64 against 2.41 ms above).
    __shared__ int2 s_buf[kLevelThreads / 32][kLevelBuffer];
    int2 *buf = s_buf[threadIdx.x >> 5];
    int kept = 0;
    auto flush = [&]() {
        __syncwarp();
        for (int k0 = 0; k0 < kept; k0 += 32) {
            const int k = k0 + lane;
            RandEntry e = {};
            uint32_t od = 0;
            if (k < kept) {
                const int2 en = buf[k];
                e = L.cur.ent[en.x];
                e.y = en.y;
                e.out_beg = (uint32_t)g.out_off[e.y];
                od = (uint32_t)g.out_off[e.y + 1] - e.out_beg;  // a node without out-edges ends here
                e.id8 = (uint32_t)g.int2ext[e.y] >> g.rec_shift;
                e.ex = walks[(int64_t)e.walk * l_max + (e.len - L.j - 3)];  // the next level's
            }
            long long item;
            const long long pos = rand_reserve(od, L.packed_out, L.check_out, &item);
            if (od > 0 && pos < L.next.cap) {
                L.next.ent[pos] = e;
                L.next.first[pos] = item;
            }
        }
        kept = 0;
        __syncwarp();
    };
    const long long *first = L.cur.first;
    for (long long t0 = warp * run; t0 < E; t0 += nwarps * run) {
        const long long t1 = min(E, t0 + run);
        // the entry of item t0: the last f with first[f] <= t0, by a 32-way search
        long long f = 0;
        for (long long span = F; span > 1;) {
            const long long step = (span + 31) / 32, at = f + lane * step;
            const unsigned le = __ballot_sync(0xffffffffu, lane * step < span && first[at] <= t0);
            const int k = 31 - __clz(le);  // lane 0 always holds
            f += k * step;
            span = min(step, span - k * step);
        }
        long long win = f + 1 + lane < F ? first[f + 1 + lane] : E;  // first items of the entries after f
        long long beg_f = first[f];
        int32_t c_y = 0, c_ex = 0, c_b = 0, c_i = 0;  // the lane's entry
        uint32_t c_k = 0, c_key = 0, c_id8 = 0;
        long long c_f = -1, c_col = 0;
        // stage 3 of an item: the draw; idx >= 0 asks for that in-list entry
        auto draw = [&](int32_t x, int4 rec) -> int32_t {
            const U32x4 d = philox4x32_10(c_k, (1u << 24) | ((uint32_t)c_i << 8) | (uint32_t)L.j, (uint32_t)rec.z, 0u,
                                          seed, c_key);
            // kept with probability sqrt(c); then the sampled in-edge (v, x) must have v = y
            const bool may = x != c_ex && d.y < t_keep && rec_may_be(rec.w, d.x, c_id8);
            return may ? rec.x + (int32_t)__umulhi(d.x, (uint32_t)rec.y) : -1;
        };
        // stage 4: members are counted at an instance's last level, else kept for the next level's list
        auto settle = [&](int32_t x, int32_t idx, int32_t v) {
            const bool member = idx >= 0 && v == c_y, last = c_i - 2 == L.j;
            if (member && last) atomicAdd(L.counts + (int64_t)c_b * g.n + x, 1);  // in H_{i-1}: the result
            const unsigned m = __ballot_sync(0xffffffffu, member && !last);
            if (m) {
                if (member && !last) buf[kept + __popc(m & ((1u << lane) - 1u))] = make_int2((int32_t)c_f, x);
                kept += __popc(m);
                if (kept > kLevelBuffer - 32) flush();
            }
        };
        for (long long t = t0; t < t1;) {
            const long long next_first = __shfl_sync(0xffffffffu, win, 0);
            int r = 0;  // entries of the window that start at or before the lane's item
            if (next_first <= t + 31) {
                const long long it = t + lane;
#pragma unroll
                for (int s = 16; s; s >>= 1) {
                    const long long v = __shfl_sync(0xffffffffu, win, r + s - 1);
                    if (v <= it) r += s;
                }
            }
            const long long start = __shfl_sync(0xffffffffu, win, r > 0 ? r - 1 : 0);
            if (f + r != c_f) {
                c_f = f + r;
                if (c_f < F) {  // past the last entry only for lanes past the last item
                    const RandEntry e = L.cur.ent[c_f];
                    c_y = e.y;
                    c_id8 = e.id8;
                    c_i = e.len;
                    c_b = e.q;
                    c_k = e.k;
                    c_key = qkey[e.q];
                    c_ex = e.ex;
                    c_col = (long long)e.out_beg - (r > 0 ? start : beg_f);
                }
            }
            const long long left = min(t1, next_first) - t;
            if (left >= 64) {  // one entry: its items in a pipeline of four stages, a load of each in flight
                const int32_t *col = g.out_col + c_col + t + lane;
                const int32_t steps = (int32_t)(left >> 5);
                int32_t x0 = __ldg(col), x1 = __ldg(col + 32), xp = 0, vp = 0, ip = -1;
                int4 r0 = __ldg(g.rec + x0);
                for (int32_t k = 0; k < steps; ++k) {
                    const int32_t x2 = k + 2 < steps ? __ldg(col + 32 * (k + 2)) : x1;
                    const int4 r1 = __ldg(g.rec + x1);
                    const int32_t idx = draw(x0, r0);
                    const int32_t v = __ldg(g.in_col + max(idx, 0));
                    settle(xp, ip, vp);
                    xp = x0, ip = idx, vp = v;
                    x0 = x1, r0 = r1, x1 = x2;
                }
                settle(xp, ip, vp);
                t += 32ll * steps;
            } else {
                const bool live = t + lane < t1;
                const int32_t x = live ? __ldg(g.out_col + c_col + t + lane) : c_ex;
                const int32_t idx = live ? draw(x, __ldg(g.rec + x)) : -1;
                settle(x, idx, __ldg(g.in_col + max(idx, 0)));
                t += 32;
            }
            // the window moves past the entries that start by item t
            const int adv = __popc(__ballot_sync(0xffffffffu, win <= t));
            if (adv > 0 && t < t1) {
                beg_f = __shfl_sync(0xffffffffu, win, adv - 1);
                f += adv;
                win = f + 1 + lane < F ? first[f + 1 + lane] : E;
            }
        }
    }
    if (kept) flush();
}

__global__ void k_rand_finalize(int32_t n, int32_t B, const int32_t *__restrict__ qnode,
                                const int32_t *__restrict__ counts, const float *__restrict__ inv_nr,
                                const int32_t *__restrict__ ext2int, float shift, float *__restrict__ out) {
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t b = blockIdx.y;
    if (v >= n) return;
    float s = (float)counts[(int64_t)b * n + ext2int[v]] * inv_nr[b] + shift;
    if ((int32_t)v == qnode[b]) s = 1.f;
    out[(int64_t)b * n + v] = s;
}

void launch_inst_init(const QueryBatch &q, const DeviceGraph &g, const int32_t *lens, int32_t w0, int32_t nw,
                      int32_t l_max, int32_t max_len, const int32_t *walks, RandList out, unsigned long long *packed,
                      unsigned long long *check, const int32_t *walk_slot, const uint8_t *t_sw, cudaStream_t s) {
    if (nw <= 0 || max_len < 2) return;
    const int64_t threads = (int64_t)nw * (max_len - 1);
    k_inst_init<<<(unsigned)((threads + 255) / 256), 256, 0, s>>>(q, g, lens, w0, nw, l_max, max_len, walks, out, packed,
                                                                  check, walk_slot, t_sw);
}
void launch_add_i32(int32_t *a, const int32_t *b, int64_t count, cudaStream_t s) {
    if (count > 0) k_add_i32<<<grid_for(count, 256, 8), 256, 0, s>>>(a, b, count);
}
void launch_rand_level(const DeviceGraph &g, const int32_t *walks, int32_t l_max, const uint32_t *qkey,
                       uint32_t seed, uint32_t t_keep, const RandLevel &L, int64_t E, cudaStream_t s) {
    const int blocks = grid_for(E, kLevelThreads, 8);
    k_rand_level<<<blocks, kLevelThreads, 0, s>>>(g, walks, l_max, qkey, seed, t_keep, L);
}
void launch_rand_finalize(int32_t n, int32_t B, const int32_t *qnode, const int32_t *counts, const float *inv_nr,
                          const int32_t *ext2int, float shift, float *out, cudaStream_t s) {
    dim3 grid((unsigned)((n + 255) / 256), (unsigned)B);
    k_rand_finalize<<<grid, 256, 0, s>>>(n, B, qnode, counts, inv_nr, ext2int, shift, out);
}

}  // namespace ps
