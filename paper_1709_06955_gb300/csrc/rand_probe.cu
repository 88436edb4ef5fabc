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
constexpr int kLevelSteps = 4;        // steps of 32 items whose loads go out together
constexpr int kLevelBuffer = 128;     // members a warp holds back before it appends them
constexpr int kLevelMaxItems = 4096;  // work items a warp takes at a time, at most

// One level.  A warp takes a run of consecutive work items (32 to kLevelMaxItems, so that a short level still spreads
// over the chip) and holds a window of 32 entries, one per lane.  A step's entry starts form a 32-bit mask (one warp
// reduction) whose set bits up to a lane count the entries to the lane's own; shuffles bring that entry's fields where
// they are used.  kLevelSteps steps go together, stage by stage -- out-edges, records, draws, in-edges -- so a warp waits
// for three gathers per 128 items, whether they belong to one hub or to a hundred short lists.
// What bounds it: dependent random sectors (a record per item; an in-list entry for a fifth of them) at 32 warps per
// SM, then the ten Philox rounds (a third of the time at level 0 went when they were left out).
// A top-k call of four queries at eps = 0.1 on R-MAT 2^20: 6.2 ms with hash sets (4.5 ms of level kernels, 0.55 ms of
// clears, two synchronisations a level); 3.0 without them; 2.3 with the records, appends gathered per warp and an entry
// load per 32 items; 1.8 with the window (its level 1, short lists: 0.55 -> 0.30 ms; level 0, 60 million items, 0.49 ->
// 0.44).  64 mixed-eps queries with the switch on R-MAT 2^22: 332 ms of level kernels with hash sets, 72 now (the call
// 97 ms; 109 at two steps, 101 at three, 114 at four with three blocks per SM).
__global__ void __launch_bounds__(kLevelThreads, 4) k_rand_level(DeviceGraph g, const int32_t *__restrict__ walks,
                                                              int32_t l_max,
                                                              const uint32_t *__restrict__ qkey, uint32_t seed,
                                                              uint32_t t_keep, RandLevel L) {
    pdl_wait();  // the level before writes the lists and the counter
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
        const int32_t n_items = (int32_t)(min(E, t0 + run) - t0);  // positions below count from t0
        // the entry of item t0: the last f with first[f] <= t0, by a 32-way search
        long long f = 0;
        for (long long span = F; span > 1;) {
            const long long step = (span + 31) / 32, at = f + lane * step;
            const unsigned le = __ballot_sync(0xffffffffu, lane * step < span && first[at] <= t0);
            const int k = 31 - __clz(le);  // lane 0 always holds
            f += k * step;
            span = min(step, span - k * step);
        }
        for (int32_t p = 0; p < n_items; f += 32) {
            // the window: entry f + lane, its start (clamped to this run) and its out-list minus its start
            RandEntry en = {};
            int32_t start = 1 << 30;
            uint32_t base = 0, key = 0;
            if (f + lane < F) {
                en = L.cur.ent[f + lane];
                const long long rel = first[f + lane] - t0;
                start = rel < 0 ? -1 : (int32_t)min(rel, (long long)(1 << 30));
                base = en.out_beg - (uint32_t)rel;
                key = qkey[en.q];
            }
            const uint32_t meta = ((uint32_t)en.len << 8) | en.id8;
            const long long wend = (f + 32 < F ? first[f + 32] : E) - t0;
            const int32_t lim = (int32_t)min((long long)n_items, wend);
            int32_t before = __popc(__ballot_sync(0xffffffffu, start < p));  // window entries that start before p
            while (p < lim) {
                int32_t x[kLevelSteps], r[kLevelSteps], idx[kLevelSteps];
                int4 rec[kLevelSteps];
#pragma unroll
                for (int u = 0; u < kLevelSteps; ++u) {
                    const int32_t q = p + 32 * u;
                    const uint32_t off = (uint32_t)(start - q);
                    const unsigned starts = __reduce_or_sync(0xffffffffu, off < 32u && q < lim ? 1u << off : 0u);
                    r[u] = (before + __popc(starts & (0xffffffffu >> (31 - lane))) - 1) & 31;
                    const uint32_t col = __shfl_sync(0xffffffffu, base, r[u]);
                    x[u] = q + lane < lim ? __ldg(g.out_col + (uint32_t)(col + q + lane)) : -1;
                    before += __popc(starts);
                }
#pragma unroll
                for (int u = 0; u < kLevelSteps; ++u) rec[u] = __ldg(g.rec + max(x[u], 0));
#pragma unroll
                for (int u = 0; u < kLevelSteps; ++u) {  // the draws
                    const uint32_t m = __shfl_sync(0xffffffffu, meta, r[u]);
                    const uint32_t k = __shfl_sync(0xffffffffu, en.k, r[u]), ky = __shfl_sync(0xffffffffu, key, r[u]);
                    const int32_t ex = __shfl_sync(0xffffffffu, en.ex, r[u]);
                    const U32x4 d = philox4x32_10(k, (1u << 24) | (m & 0xFFFFFF00u) | (uint32_t)L.j, (uint32_t)rec[u].z,
                                                  0u, seed, ky);
                    // kept with probability sqrt(c); then the sampled in-edge (v, x) must have v = y
                    const bool may = x[u] >= 0 && x[u] != ex && d.y < t_keep && rec_may_be(rec[u].w, d.x, m & 0xFFu);
                    idx[u] = may ? rec[u].x + (int32_t)__umulhi(d.x, (uint32_t)rec[u].y) : -1;
                }
                int32_t v[kLevelSteps];
#pragma unroll
                for (int u = 0; u < kLevelSteps; ++u) v[u] = idx[u] >= 0 ? __ldg(g.in_col + idx[u]) : -1;
#pragma unroll
                for (int u = 0; u < kLevelSteps; ++u) {
                    const int32_t y = __shfl_sync(0xffffffffu, en.y, r[u]);
                    const bool member = v[u] == y && idx[u] >= 0;
                    if (!__any_sync(0xffffffffu, member)) continue;
                    // members are counted at an instance's last level, else kept for the next level's list
                    const bool last = (int32_t)(__shfl_sync(0xffffffffu, meta, r[u]) >> 8) - 2 == L.j;
                    if (member && last) atomicAdd(L.counts + (int64_t)L.cur.ent[f + r[u]].q * g.n + x[u], 1);
                    const unsigned m = __ballot_sync(0xffffffffu, member && !last);
                    if (m) {
                        if (member && !last)
                            buf[kept + __popc(m & ((1u << lane) - 1u))] = make_int2((int32_t)(f + r[u]), x[u]);
                        kept += __popc(m);
                        if (kept > kLevelBuffer - 32) flush();
                    }
                }
                p = min(lim, p + 32 * kLevelSteps);
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
    pdl_launch(k_rand_level, dim3(blocks), dim3(kLevelThreads), 0, s, g, walks, l_max, qkey, seed, t_keep, L);
}
void launch_rand_finalize(int32_t n, int32_t B, const int32_t *qnode, const int32_t *counts, const float *inv_nr,
                          const int32_t *ext2int, float shift, float *out, cudaStream_t s) {
    dim3 grid((unsigned)((n + 255) / 256), (unsigned)B);
    k_rand_finalize<<<grid, 256, 0, s>>>(n, B, qnode, counts, inv_nr, ext2int, shift, out);
}

}  // namespace ps
