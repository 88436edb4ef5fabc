// Device-side update of the graph store: one batch of edge insertions or deletions merged into the CSR
// arrays without rebuilding them on the host.
//
// The batch comes deduplicated, without loops and in two orders, sorted on the device (graph_build.cu's radix sort): by
// (destination, source in the caller's id order) for the in-lists, whose order is the caller's source-id order (walks
// pick the k-th entry of it), and by (source, destination in internal id order) for the out-lists.  Then the kernels
// below
//   1. marks the batch entries that change the graph (an insert of an absent edge, a delete of a present one)
//      by binary search in the current rows, and counts the change of every row's degree;
//   2. forms the new offsets (prefix sums of the new degrees);
//   3. writes the rows: an old entry that survives moves by its row's distance plus the number of inserted entries
//      ordered before it in the row, minus the number of deleted ones; an inserted entry goes to the number of old
//      entries ordered before it plus its rank among the inserts
//   4. recomputes w[v] = sqrt(c)/|I(v)| and the pull pieces (a counting sort by piece length).
#include <algorithm>

#include "internal.cuh"

namespace ps {

struct UpdateBatch {
    int64_t k = 0;
    // in-order: sorted by (dst internal, src external)
    const int32_t *in_dst = nullptr, *in_src = nullptr, *in_src_ext = nullptr;
    // out-order: sorted by (src internal, dst internal)
    const int32_t *out_src = nullptr, *out_dst = nullptr;
    long long *in_valid = nullptr, *out_valid = nullptr;  // 1 if the entry changes the graph
    const long long *in_vpre = nullptr, *out_vpre = nullptr;  // exclusive prefix sums of the flags (k + 1)
    bool insert = true;
};

// first index in [lo, hi) of row entries whose key is >= x, keys read through `key`
template <class Key>
__device__ __forceinline__ int64_t lower_bound_row(int64_t lo, int64_t hi, uint32_t x, Key key) {
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (key(mid) < x) lo = mid + 1; else hi = mid;
    }
    return lo;
}

// 1. validity of each batch entry (in-order and out-order copies get the same decision) and degree deltas
__global__ void k_upd_mark(DeviceGraph g, UpdateBatch b, long long *in_delta, long long *out_delta) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= b.k) return;
    {
        const int32_t v = b.in_dst[e];
        const uint32_t xe = (uint32_t)b.in_src_ext[e];
        const int64_t beg = g.in_off[v], end = g.in_off[v + 1];
        const int64_t pos = lower_bound_row(beg, end, xe, [&](int64_t i) { return (uint32_t)g.int2ext[g.in_col[i]]; });
        const bool exists = pos < end && (uint32_t)g.int2ext[g.in_col[pos]] == xe;
        const bool valid = b.insert ? !exists : exists;
        b.in_valid[e] = valid ? 1 : 0;
        if (valid) atomicAdd(reinterpret_cast<unsigned long long *>(&in_delta[v]), b.insert ? 1ull : ~0ull);  // +-1
    }
    {
        const int32_t x = b.out_src[e];
        const uint32_t v = (uint32_t)b.out_dst[e];
        const int64_t beg = g.out_off[x], end = g.out_off[x + 1];
        const int64_t pos = lower_bound_row(beg, end, v, [&](int64_t i) { return (uint32_t)g.out_col[i]; });
        const bool exists = pos < end && (uint32_t)g.out_col[pos] == v;
        const bool valid = b.insert ? !exists : exists;
        b.out_valid[e] = valid ? 1 : 0;
        if (valid) atomicAdd(reinterpret_cast<unsigned long long *>(&out_delta[x]), b.insert ? 1ull : ~0ull);
    }
}

// new degree per row
__global__ void k_upd_degrees(int32_t n, const int64_t *__restrict__ off, const long long *__restrict__ delta,
                              long long *deg) {
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v < n) deg[v] = (off[v + 1] - off[v]) + delta[v];
}

// 3a. The batch entries' rows as boundaries of the old list: [beg, end) of the entry's row, the first batch entry of the
// row, and the distance by which the row and what follows it move.
struct RowBound {
    long long beg, end, first, shift, shift_after;
};
__global__ void k_upd_bounds(int64_t k, const int32_t *__restrict__ rows, const int64_t *__restrict__ off,
                             const long long *__restrict__ new_off, RowBound *out) {
    const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (e >= k) return;
    const int32_t r = rows[e];
    int64_t lo = 0, hi = e;  // the first entry of row r
    while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if (rows[mid] < r) lo = mid + 1; else hi = mid;
    }
    const long long beg = off[r], end = off[r + 1];
    out[e] = RowBound{beg, end, lo, new_off[r] - beg, new_off[r + 1] - end};
}

// 3b. The old entries: a warp per kMoveTile of them, whatever rows they belong to, so neither a hub's row nor many short
// rows leave lanes idle.  Between two touched rows everything moves by one distance, a plain copy; in a touched row the
// valid batch entries before an entry are counted with a binary search in the row's batch range and the prefix sums of
// the validity flags.  Keys compare in the row's order: the caller's source id for in-lists, the internal destination id
// for out-lists.  What bounds it: reading and writing the list.  Two batches of 10,000 edges and a query on R-MAT 2^21
// took 10.9 ms with a warp per row, which searched the batch for every row (1.4 ms a list); 5.6 ms by tiles (0.08 to
// 0.2 ms a list).  Rows of fewer than 32 entries in a row of touched ones are taken 32 entries at a time, each lane
// finding its own: inserted edges of nodes that had none leave thousands of such rows side by side (1.6 ms a list
// without that).
constexpr int kMoveTile = 2048;
template <bool IN>
__global__ void __launch_bounds__(256) k_upd_move(DeviceGraph g, UpdateBatch b, const RowBound *__restrict__ bound,
                                                  int32_t *__restrict__ new_col) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
    const long long *valid = IN ? b.in_valid : b.out_valid;
    const long long *vpre = IN ? b.in_vpre : b.out_vpre;
    const int32_t *col = IN ? g.in_col : g.out_col;
    int64_t pos = warp * kMoveTile;
    const int64_t end = min(g.m, pos + kMoveTile);
    // old entry i in the touched row of boundary q, whose batch entries are rb.first .. q
    auto move_one = [&](int64_t i, int64_t q, const RowBound &rb) {
        auto bkey = [&](int64_t j) -> uint32_t { return IN ? (uint32_t)b.in_src_ext[j] : (uint32_t)b.out_dst[j]; };
        const int32_t c = col[i];
        const uint32_t x = IN ? (uint32_t)g.int2ext[c] : (uint32_t)c;
        const int64_t j = lower_bound_row(rb.first, q + 1, x, bkey);  // first batch entry with key >= x
        if (!b.insert && j <= q && bkey(j) == x && valid[j]) return;  // deleted
        const long long less = vpre[j] - vpre[rb.first];
        new_col[i + rb.shift + (b.insert ? less : -less)] = c;
    };
    int64_t e = -1;  // the last boundary that starts at or before pos
    while (pos < end) {
        for (int64_t span = b.k - e; span > 1;) {  // 32-way search
            const int64_t step = (span + 31) / 32, at = e + lane * step;
            const unsigned le = __ballot_sync(0xffffffffu, lane * step < span && (at < 0 || bound[at].beg <= pos));
            const int j = 31 - __clz(le);  // lane 0 always holds
            e += j * step;
            span = min(step, span - j * step);
        }
        RowBound rb = {0, 0, 0, 0, 0};
        if (e >= 0) rb = bound[e];
        const bool touched = e >= 0 && pos < rb.end;
        const int64_t stop = min(end, touched ? (int64_t)rb.end : (e + 1 < b.k ? (int64_t)bound[e + 1].beg : g.m));
        if (stop - pos < 32 && stop < end) {  // short rows: every lane finds its own
            const int64_t i = pos + lane;
            if (i < end) {
                int64_t lo = e, hi = min(b.k, e + 33);  // 32 entries of the list lie in at most 32 more non-empty rows,
                if (hi < b.k && bound[hi].beg <= i) hi = b.k;  // but repeats and empty rows may stand between
                while (hi - lo > 1) {
                    const int64_t mid = (lo + hi) >> 1;
                    if (bound[mid].beg <= i) lo = mid; else hi = mid;
                }
                RowBound mine = {0, 0, 0, 0, 0};
                if (lo >= 0) mine = bound[lo];
                if (lo >= 0 && i < mine.end) move_one(i, lo, mine);
                else new_col[i + mine.shift_after] = col[i];
            }
            pos = min(end, pos + 32);
            continue;
        }
        if (touched) {
            for (int64_t i = pos + lane; i < stop; i += 32) move_one(i, e, rb);
        } else {
            const long long shift = rb.shift_after;
            for (int64_t i = pos + lane; i < stop; i += 128) {
                int32_t c[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) c[u] = i + 32 * u < stop ? __ldg(col + i + 32 * u) : 0;
#pragma unroll
                for (int u = 0; u < 4; ++u)
                    if (i + 32 * u < stop) new_col[i + 32 * u + shift] = c[u];
            }
        }
        pos = stop;
    }
}

// 3c. The inserted entries, a thread each.
template <bool IN>
__global__ void __launch_bounds__(256) k_upd_insert(DeviceGraph g, UpdateBatch b, const RowBound *__restrict__ bound,
                                                    int32_t *__restrict__ new_col) {
    const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (j >= b.k || !(IN ? b.in_valid : b.out_valid)[j]) return;
    const long long *vpre = IN ? b.in_vpre : b.out_vpre;
    const int32_t *col = IN ? g.in_col : g.out_col;
    const RowBound rb = bound[j];
    const uint32_t x = IN ? (uint32_t)b.in_src_ext[j] : (uint32_t)b.out_dst[j];
    const int64_t at = lower_bound_row(rb.beg, rb.end, x, [&](int64_t i) -> uint32_t {
        return IN ? (uint32_t)g.int2ext[col[i]] : (uint32_t)col[i];
    });
    new_col[at + rb.shift + (vpre[j] - vpre[rb.first])] = IN ? b.in_src[j] : b.out_dst[j];
}

// 4. w, the node records and the pull pieces (offsets fit 32 bits: m < 2^31)
__global__ void k_upd_w(int32_t n, const long long *__restrict__ new_off, const int32_t *__restrict__ in_col,
                        float sqrt_c, const int32_t *__restrict__ int2ext, int32_t rec_shift, float *w, int4 *rec,
                        long long *npieces) {
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v >= n) return;
    const long long beg = new_off[v], d = new_off[v + 1] - beg;
    w[v] = d > 0 ? sqrt_c / (float)d : 0.f;
    uint32_t splits = 0;
    if (d > 0) {
        int32_t x[kRecSplits];
        for (int k = 0; k < kRecSplits; ++k) x[k] = in_col[beg + (k + 1) * d / (kRecSplits + 1)];
        for (int k = 0; k < kRecSplits; ++k) splits |= (uint32_t)(int2ext[x[k]] >> rec_shift) << (8 * k);
    }
    rec[v] = make_int4((int32_t)beg, (int32_t)d, int2ext[v], (int32_t)splits);
    npieces[v] = d <= kPiece ? 1 : (d + kPiece - 1) / kPiece;
}

// Pull pieces, a counting sort by (row has out-edges first, then length, longest first): the pieces of the rows that
// somebody reads (below *n_active) come first, so a pull whose result is only gathered runs over them alone.  Bucket of
// a piece: length for an active row, kPiece + 1 + length for another.  A block takes a range of rows and counts in shared
// memory; with one global counter per length a million rows queued on a few hot counters (R-MAT 2^21: 0.81 and 1.01 ms
// for the two passes, now 0.01 and 0.12).
constexpr int kPieceBuckets = 2 * (kPiece + 1);
constexpr int kPieceThreads = 256;

__device__ __forceinline__ void piece_counts(long long d, bool active, int *full, int *rest, int *fb, int *rb) {
    const int base = active ? 0 : kPiece + 1;
    *full = d <= kPiece ? 0 : (int)(d / kPiece);
    *rest = d <= kPiece ? 1 : (d % kPiece != 0);
    *fb = base + kPiece;
    *rb = base + (d <= kPiece ? (int)d : (int)(d % kPiece));
}

__global__ void __launch_bounds__(kPieceThreads) k_upd_piece_hist(int32_t n, const long long *__restrict__ new_off,
                                                                  const int32_t *__restrict__ n_active,
                                                                  unsigned long long *hist, int32_t *split_v,
                                                                  unsigned long long *n_split) {
    __shared__ unsigned s_h[kPieceBuckets];
    for (int i = threadIdx.x; i < kPieceBuckets; i += kPieceThreads) s_h[i] = 0;
    __syncthreads();
    const int64_t per = ((int64_t)n + gridDim.x - 1) / gridDim.x;
    const int64_t beg = blockIdx.x * per, end = min((int64_t)n, beg + per);
    const int32_t act = *n_active;
    for (int64_t v = beg + threadIdx.x; v < end; v += kPieceThreads) {
        const long long d = new_off[v + 1] - new_off[v];
        int full, rest, fb, rb;
        piece_counts(d, v < act, &full, &rest, &fb, &rb);
        if (full) {
            atomicAdd(&s_h[fb], (unsigned)full);
            split_v[atomicAdd(n_split, 1ull)] = (int32_t)v;
        }
        if (rest) atomicAdd(&s_h[rb], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kPieceBuckets; i += kPieceThreads)
        if (s_h[i]) atomicAdd(&hist[i], (unsigned long long)s_h[i]);
}

// bucket starts: active rows' pieces longest first, then the others'
__global__ void k_upd_piece_starts(const unsigned long long *hist, unsigned long long *cursor) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    unsigned long long acc = 0;
    for (int c = 0; c < 2; ++c)
        for (int len = kPiece; len >= 0; --len) {
            cursor[c * (kPiece + 1) + len] = acc;
            acc += hist[c * (kPiece + 1) + len];
        }
}

__global__ void __launch_bounds__(kPieceThreads) k_upd_piece_fill(int32_t n, const long long *__restrict__ new_off,
                                                                  const int32_t *__restrict__ n_active,
                                                                  unsigned long long *cursor, int32_t *pv, int64_t *pb,
                                                                  int32_t *pl) {
    __shared__ unsigned s_h[kPieceBuckets];
    __shared__ unsigned long long s_at[kPieceBuckets];
    for (int i = threadIdx.x; i < kPieceBuckets; i += kPieceThreads) s_h[i] = 0;
    __syncthreads();
    const int64_t per = ((int64_t)n + gridDim.x - 1) / gridDim.x;
    const int64_t beg = blockIdx.x * per, end = min((int64_t)n, beg + per);
    const int32_t act = *n_active;
    for (int64_t v = beg + threadIdx.x; v < end; v += kPieceThreads) {
        int full, rest, fb, rb;
        piece_counts(new_off[v + 1] - new_off[v], v < act, &full, &rest, &fb, &rb);
        if (full) atomicAdd(&s_h[fb], (unsigned)full);
        if (rest) atomicAdd(&s_h[rb], 1u);
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kPieceBuckets; i += kPieceThreads) {
        if (s_h[i]) s_at[i] = atomicAdd(&cursor[i], (unsigned long long)s_h[i]);
        s_h[i] = 0;  // each row's places are counted off again
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    for (int64_t v = beg + threadIdx.x; v < end; v += kPieceThreads) {
        const int64_t left = end - (v - lane);  // rows of this round from the warp's first on
        const unsigned lanes = left >= 32 ? 0xffffffffu : (1u << left) - 1u;
        const long long b0 = new_off[v], d = new_off[v + 1] - b0;
        int full, rest, fb, rb;
        piece_counts(d, v < act, &full, &rest, &fb, &rb);
        unsigned long long i0 = 0;
        if (full) i0 = s_at[fb] + atomicAdd(&s_h[fb], (unsigned)full);
        for (unsigned hubs = __ballot_sync(lanes, full > 0); hubs; hubs &= hubs - 1) {  // a hub's pieces by the warp
            const int src = __ffs(hubs) - 1;
            const int cnt = __shfl_sync(lanes, full, src);
            const unsigned long long at = __shfl_sync(lanes, i0, src);
            const long long hb = __shfl_sync(lanes, b0, src);
            const int32_t hv = __shfl_sync(lanes, (int32_t)v, src);
            for (int c = __popc(lanes & ((1u << lane) - 1u)); c < cnt; c += __popc(lanes)) {
                pv[at + c] = hv;
                pb[at + c] = hb + (long long)c * kPiece;
                pl[at + c] = kPiece | (int32_t)0x80000000;
            }
        }
        if (rest) {
            const unsigned long long i = s_at[rb] + atomicAdd(&s_h[rb], 1u);
            pv[i] = (int32_t)v;
            pb[i] = b0 + (long long)full * kPiece;
            pl[i] = d <= kPiece ? (int32_t)d : ((int32_t)(d % kPiece) | (int32_t)0x80000000);
        }
    }
}

static unsigned blocks_for(int64_t work, int threads) { return (unsigned)((work + threads - 1) / threads); }

void launch_upd_mark(const DeviceGraph &g, const UpdateBatchArgs &a, long long *in_delta, long long *out_delta,
                     cudaStream_t s) {
    if (a.k <= 0) return;
    UpdateBatch b;
    b.k = a.k; b.in_dst = a.in_dst; b.in_src = a.in_src; b.in_src_ext = a.in_src_ext; b.out_src = a.out_src;
    b.out_dst = a.out_dst; b.in_valid = a.in_valid; b.out_valid = a.out_valid; b.insert = a.insert;
    b.in_vpre = a.in_vpre; b.out_vpre = a.out_vpre;
    k_upd_mark<<<blocks_for(a.k, 256), 256, 0, s>>>(g, b, in_delta, out_delta);
}

void launch_upd_degrees(int32_t n, const int64_t *off, const long long *delta, long long *deg, cudaStream_t s) {
    k_upd_degrees<<<blocks_for(n, 256), 256, 0, s>>>(n, off, delta, deg);
}

size_t upd_bounds_bytes(int64_t k) { return sizeof(RowBound) * (size_t)k; }

void launch_upd_rows(const DeviceGraph &g, const UpdateBatchArgs &a, bool in_lists, const long long *new_off,
                     int32_t *new_col, void *bounds, cudaStream_t s) {
    if (a.k <= 0) return;
    UpdateBatch b;
    b.k = a.k; b.in_dst = a.in_dst; b.in_src = a.in_src; b.in_src_ext = a.in_src_ext; b.out_src = a.out_src;
    b.out_dst = a.out_dst; b.in_valid = a.in_valid; b.out_valid = a.out_valid; b.insert = a.insert;
    b.in_vpre = a.in_vpre; b.out_vpre = a.out_vpre;
    RowBound *bd = static_cast<RowBound *>(bounds);
    k_upd_bounds<<<blocks_for(a.k, 256), 256, 0, s>>>(a.k, in_lists ? a.in_dst : a.out_src,
                                                      in_lists ? g.in_off : g.out_off, new_off, bd);
    const unsigned mb = blocks_for((g.m + kMoveTile - 1) / kMoveTile * 32, 256);
    if (mb > 0 && in_lists) k_upd_move<true><<<mb, 256, 0, s>>>(g, b, bd, new_col);
    if (mb > 0 && !in_lists) k_upd_move<false><<<mb, 256, 0, s>>>(g, b, bd, new_col);
    if (!a.insert) return;
    if (in_lists) k_upd_insert<true><<<blocks_for(a.k, 256), 256, 0, s>>>(g, b, bd, new_col);
    else k_upd_insert<false><<<blocks_for(a.k, 256), 256, 0, s>>>(g, b, bd, new_col);
}

void launch_upd_w(int32_t n, const long long *new_off, const int32_t *in_col, float sqrt_c, const int32_t *int2ext,
                  int32_t rec_shift, float *w, int4 *rec, long long *npieces, cudaStream_t s) {
    k_upd_w<<<blocks_for(n, 256), 256, 0, s>>>(n, new_off, in_col, sqrt_c, int2ext, rec_shift, w, rec, npieces);
}

void launch_upd_pieces(int32_t n, const long long *new_off, const int32_t *n_active, unsigned long long *hist,
                       unsigned long long *cursor, int32_t *split_v, unsigned long long *n_split, int32_t *pv,
                       int64_t *pb, int32_t *pl, cudaStream_t s) {
    cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * kPieceBuckets, s);
    cudaMemsetAsync(n_split, 0, sizeof(unsigned long long), s);
    const int blocks = grid_for(n, 4 * kPieceThreads, 4);
    k_upd_piece_hist<<<blocks, kPieceThreads, 0, s>>>(n, new_off, n_active, hist, split_v, n_split);
    k_upd_piece_starts<<<1, 32, 0, s>>>(hist, cursor);
    k_upd_piece_fill<<<blocks, kPieceThreads, 0, s>>>(n, new_off, n_active, cursor, pv, pb, pl);
}

}  // namespace ps
