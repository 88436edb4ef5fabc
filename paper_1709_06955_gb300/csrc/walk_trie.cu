// sqrt(c)-walks (Def. 3, Pruning Rule 1), the reverse-reachability tree of Alg. 4 as a hash table, and
// the level schedule derived from it.
#include "internal.cuh"

namespace ps {

// Which query of the launch walk `wid` belongs to (walk_base is sorted, B is small).
__device__ __forceinline__ int32_t query_of(const int32_t *walk_base, int32_t B, int32_t wid) {
    int32_t lo = 0, hi = B;  // walk_base[lo] <= wid < walk_base[hi]
    while (hi - lo > 1) {
        const int32_t mid = (lo + hi) >> 1;
        if (walk_base[mid] <= wid) lo = mid; else hi = mid;
    }
    return lo;
}

// One thread per walk, in internal node ids.  At node v: stop when the draw x0 is below t_stop (probability 1 - sqrt(c)),
// stop when |I(v)| = 0, stop when the walk already holds l_max nodes; otherwise move to entry
// floor(x1 * |I(v)| / 2^32) of I(v).
__global__ void __launch_bounds__(256) k_walks(const int64_t *__restrict__ in_off, const int32_t *__restrict__ in_col,
                                               const int32_t *__restrict__ ext2int, QueryBatch q, int32_t W, int32_t l_max, uint32_t t_stop,
                                               uint32_t seed, int32_t *__restrict__ walks,
                                               int32_t *__restrict__ lens, bool pad, LaunchCounters *ctr) {
    const int32_t wid = blockIdx.x * blockDim.x + threadIdx.x;
    int32_t len = 0;
    if (wid < W) {
        const int32_t b = query_of(q.walk_base, q.B, wid);
        const uint32_t k = (uint32_t)(q.walk_k0[b] + (wid - q.walk_base[b]));
        const uint32_t key1 = q.qid[b];
        int32_t v = ext2int[q.node[b]];
        int32_t *row = walks + (int64_t)wid * l_max;
        row[len++] = v;
        for (uint32_t s = 0;; ++s) {
            if (len >= l_max) break;
            const U32x4 r = philox4x32_10(k, s, 0u, 0u, seed, key1);
            if (r.x < t_stop) break;
            const int64_t beg = in_off[v];
            const uint32_t d = (uint32_t)(in_off[v + 1] - beg);
            if (d == 0) break;
            v = in_col[beg + __umulhi(r.y, d)];
            row[len++] = v;
        }
        if (pad)
            for (int32_t t = len; t < l_max; ++t) row[t] = -1;
        lens[wid] = len;
    }
    // block-level reduction of the length sum and maximum
    __shared__ unsigned long long s_sum[8];
    __shared__ int32_t s_max[8];
    unsigned long long sum = (unsigned long long)len;
    int32_t mx = len;
    for (int o = 16; o; o >>= 1) {
        sum += __shfl_xor_sync(0xffffffffu, sum, o);
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) { s_sum[warp] = sum; s_max[warp] = mx; }
    __syncthreads();
    if (threadIdx.x == 0) {
        unsigned long long bs = 0;
        int32_t bm = 0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) { bs += s_sum[i]; bm = max(bm, s_max[i]); }
        atomicAdd(&ctr->walk_nodes, bs);
        atomicMax(&ctr->max_len, bm);
    }
}

void launch_walks(const DeviceGraph &g, const QueryBatch &q, int32_t W, int32_t l_max, uint32_t t_stop,
                  uint32_t seed, int32_t *walks, int32_t *lens, bool pad, LaunchCounters *ctr, cudaStream_t s) {
    if (W <= 0) return;
    k_walks<<<(W + 255) / 256, 256, 0, s>>>(g.in_off, g.in_col, g.ext2int, q, W, l_max, t_stop, seed, walks, lens, pad, ctr);
}

// splitmix64 finalizer as the table hash
__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Returns the slot holding `key`, inserting it if absent; -1 when the table is full (every probe is
// bounded by the capacity, so the loop always ends).
__device__ __forceinline__ int64_t table_insert(unsigned long long *keys, int64_t cap, unsigned long long key) {
    int64_t h = (int64_t)(mix64(key) & (unsigned long long)(cap - 1));
    for (int64_t probe = 0; probe < cap; ++probe) {
        unsigned long long cur = keys[h];
        if (cur == key) return h;
        if (cur == kEmptyKey) {
            cur = atomicCAS(&keys[h], kEmptyKey, key);
            if (cur == kEmptyKey || cur == key) return h;
        }
        h = (h + 1) & (cap - 1);
    }
    return -1;
}

// One thread per walk: inserts the super-root, then the prefixes (u_1), (u_1,u_2), ... (Alg. 4 lines
// 5-11).  A node's weight counts the walks through it; its height is the longest walk suffix below it.
__global__ void __launch_bounds__(256) k_trie_insert(QueryBatch q, int32_t W, int32_t l_max,
                                                     const int32_t *__restrict__ walks,
                                                     const int32_t *__restrict__ lens, TrieTable t,
                                                     LaunchCounters *ctr) {
    const int32_t wid = blockIdx.x * blockDim.x + threadIdx.x;
    if (wid >= W) return;
    const int32_t b = query_of(q.walk_base, q.B, wid);
    const int32_t len = lens[wid];
    const int32_t *row = walks + (int64_t)wid * l_max;
    int64_t p = table_insert(t.key, t.cap, ((unsigned long long)kRhoTag << 32) | (uint32_t)b);
    if (p < 0) { atomicExch(&ctr->overflow, 1); return; }
    t.node[p] = -1;
    t.parent[p] = -1;
    t.depth[p] = 0;
    t.query[p] = b;
    atomicMax(&t.height[p], len);
    for (int32_t i = 1; i <= len; ++i) {
        const int32_t u = row[i - 1];
        const int64_t s = table_insert(t.key, t.cap, ((unsigned long long)(uint32_t)p << 32) | (uint32_t)u);
        if (s < 0) { atomicExch(&ctr->overflow, 1); return; }
        if (t.walk_slot) t.walk_slot[(int64_t)wid * l_max + i - 1] = (int32_t)s;
        t.node[s] = u;
        t.parent[s] = (int32_t)p;
        t.depth[s] = i;
        t.query[s] = b;
        const int32_t through = atomicAdd(&t.weight[s], 1);
        atomicMax(&t.height[s], len - i);
        if (t.probes && through == 0 && i >= 2) {  // the first walk through a prefix lists it as a probe
            const unsigned mask = __activemask();
            const int lane = threadIdx.x & 31, leader = __ffs(mask) - 1;
            int32_t base = 0;
            if (lane == leader) base = atomicAdd(t.probe_count, __popc(mask));
            base = __shfl_sync(mask, base, leader);
            t.probes[base + __popc(mask & ((1u << lane) - 1u))] = (int32_t)s;
        }
        p = s;
    }
}

void launch_trie_insert(const DeviceGraph &g, const QueryBatch &q, int32_t W, int32_t l_max, const int32_t *walks,
                        const int32_t *lens, TrieTable t, LaunchCounters *ctr, cudaStream_t s) {
    (void)g;
    if (W <= 0) return;
    k_trie_insert<<<(W + 255) / 256, 256, 0, s>>>(q, W, l_max, walks, lens, t, ctr);
}

// ------------------------------------------------------------------------------------------------
// level schedule: two passes over the tree's table.  The first counts the nodes of each depth by class -- without a column,
// dense (height >= 3, and a super-root of height 2), push (height 2) -- and leaves the class in the slot; the second
// writes every node into its depth's list and exports the nodes that own a column (dense or push).  Both count in shared
// memory and take one global add per block and counter: the counters are a few dozen addresses that every node would
// queue on.  The export goes straight to the host's pinned memory, so one synchronisation brings the counts and the nodes.
// (R-MAT 2^18, two queries at eps 0.05, 59,404 nodes: 46 us in three kernels, 19 in these two.)
// ------------------------------------------------------------------------------------------------
constexpr int kSchedThreads = 256, kSchedPer = 4;

// count: [3][D1]
__global__ void __launch_bounds__(kSchedThreads) k_sched_count(TrieTable t, int32_t D1, int32_t *count) {
    extern __shared__ int32_t sh[];
    for (int i = threadIdx.x; i < 3 * D1; i += kSchedThreads) sh[i] = 0;
    __syncthreads();
    const int64_t e0 = blockIdx.x * (int64_t)(kSchedThreads * kSchedPer) + threadIdx.x;
#pragma unroll
    for (int u = 0; u < kSchedPer; ++u) {
        const int64_t e = e0 + u * kSchedThreads;
        if (e >= t.cap || t.key[e] == kEmptyKey) continue;
        const int32_t d = t.depth[e], h = t.height[e];
        const int cls = h >= 3 || (d == 0 && h >= 2) ? 1 : (h == 2 ? 2 : 0);
        t.slot[e] = cls == 1 ? 0 : (cls == 2 ? -2 : -1);
        atomicAdd(&sh[cls * D1 + d], 1);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < 3 * D1; i += kSchedThreads)
        if (sh[i] > 0) atomicAdd(&count[i], sh[i]);
}

// cur: [D1 + 1], zero; cur[D1] counts the exported nodes.  out: three arrays of `stride`: entry, parent entry (-1 - query
// at depth 0), 2 * depth + (1 if dense).
__global__ void __launch_bounds__(kSchedThreads) k_sched_lists(TrieTable t, int32_t D1, const int32_t *__restrict__ count,
                                                               int32_t *cur, int32_t *node_list, int32_t *out,
                                                               int64_t stride) {
    extern __shared__ int32_t sh[];
    int32_t *s_n = sh, *s_at = sh + D1 + 1;
    for (int i = threadIdx.x; i <= D1; i += kSchedThreads) s_n[i] = 0;
    __syncthreads();
    const int64_t e0 = blockIdx.x * (int64_t)(kSchedThreads * kSchedPer) + threadIdx.x;
    int32_t dep[kSchedPer], pos[kSchedPer], slot[kSchedPer], at[kSchedPer];
#pragma unroll
    for (int u = 0; u < kSchedPer; ++u) {
        const int64_t e = e0 + u * kSchedThreads;
        dep[u] = -1;
        if (e >= t.cap || t.key[e] == kEmptyKey) continue;
        dep[u] = t.depth[e];
        slot[u] = t.slot[e];
        pos[u] = atomicAdd(&s_n[dep[u]], 1);
        if (slot[u] != -1) at[u] = atomicAdd(&s_n[D1], 1);
    }
    __syncthreads();
    if (threadIdx.x < 32) {  // the depths' offsets, and this block's place in each
        int32_t base = 0;
        for (int d0 = 0; d0 <= D1; d0 += 32) {
            const int d = d0 + threadIdx.x;
            int32_t x = d < D1 ? count[d] + count[D1 + d] + count[2 * D1 + d] : 0, sum = x;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int32_t y = __shfl_up_sync(0xffffffffu, sum, o);
                if ((int)threadIdx.x >= o) sum += y;
            }
            if (d <= D1) s_at[d] = (d < D1 ? base + sum - x : 0) + (s_n[d] > 0 ? atomicAdd(&cur[d], s_n[d]) : 0);
            base += __shfl_sync(0xffffffffu, sum, 31);
        }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kSchedPer; ++u) {
        if (dep[u] < 0) continue;
        const int64_t e = e0 + u * kSchedThreads;
        node_list[s_at[dep[u]] + pos[u]] = (int32_t)e;
        if (slot[u] == -1) continue;
        const int64_t i = s_at[D1] + at[u];
        out[i] = (int32_t)e;
        out[stride + i] = dep[u] > 0 ? t.parent[e] : -1 - t.query[e];
        out[2 * stride + i] = 2 * dep[u] + (slot[u] >= 0 ? 1 : 0);
    }
}

void launch_sched(TrieTable t, int32_t D1, int32_t *count, int32_t *cur, int32_t *node_list, int32_t *out, int64_t stride,
                  cudaStream_t s) {
    const unsigned blocks = (unsigned)((t.cap + kSchedThreads * kSchedPer - 1) / (kSchedThreads * kSchedPer));
    k_sched_count<<<blocks, kSchedThreads, 3 * D1 * sizeof(int32_t), s>>>(t, D1, count);
    k_sched_lists<<<blocks, kSchedThreads, 2 * (D1 + 1) * sizeof(int32_t), s>>>(t, D1, count, cur, node_list, out, stride);
}

// slot[ent[i]] = col[i]
__global__ void k_set_slots(TrieTable t, const int32_t *__restrict__ ent, const int32_t *__restrict__ col, int32_t count) {
    const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < count) t.slot[ent[i]] = col[i];
}

void launch_set_slots(TrieTable t, const int32_t *ent, const int32_t *col, int32_t count, cudaStream_t s) {
    if (count > 0) k_set_slots<<<(count + 255) / 256, 256, 0, s>>>(t, ent, col, count);
}

}  // namespace ps
