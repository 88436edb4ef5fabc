// PROBE level loop over the reverse-reachability tree (Alg. 2 / Alg. 4), regrouped.
//
// Alg. 4 probes every tree node r_q (the prefix (u_1..u_q)) with q-1 levels of Alg. 2 and adds
// w_q/n_r * PROBE(u_1..u_q).  Writing one level of Alg. 2 as a linear map, Score_{j+1} = X_a M Score_j
// with (M y)[v] = sqrt(c)/|I(v)| * sum_{x in I(v)} y[x] and X_a zeroing entry a = u_{q-j-1}, the sum over
// all tree nodes factors along the tree (Horner's rule): for a tree node t with graph node a,
//     C(t)  = sum over children s of Y(s),        Y(s) = w_s/n_r e_{a_s} + X_{a_s} M C(s),
// and the estimate is M C(root) (entry u then set to 1).  Because X_a only removes entry a,
//     X_a M C = M C - beta e_a,   beta = (M C)[a] = sqrt(c)/|I(a)| * sum_{x in I(a)} C[x],
// so with gamma_s = w_s/n_r - beta_s the children of one tree node share one application of M:
//     C(t) = M D(t) + sum_s gamma_s e_{a_s},  D(t) = sum over children s of C(s).
// A tree node whose subtree has height >= 2 owns a score vector MD(t) = M D(t) (a column); lower nodes
// only contribute their sparse gamma terms.  For height >= 3 the column is "dense" and computed by the
// pull; for height 2, D(t) is just the gamma terms of t's grandchildren (all leaves), so the column is
// "pushed": MD(t) = sum_g gamma_g * sum_{x in O(a_g)} sqrt(c)/|I(x)| e_x.  The level loop runs from the
// deepest depth to the virtual super-root (depth 0, whose only child is the root u):
//   accumulate D(t)[x] = sum of the children's MD columns, in place      (dense t; an heir's column is reused)
//   scatter  D(t)[a_g] += gamma_g for every grandchild g of t            (sparse terms, dense t)
//   pull     MD(t)[v] = sqrt(c)/|I(v)| * sum_{x in I(v)} D(t)[x]         (the dominant kernel, dense t)
//   push     MD(t)[x] += sqrt(c)/|I(x)| * gamma_g, x in O(a_g)           (height-2 t)
//   gamma    gamma_t  = w_t/n_r - sqrt(c)/|I(a_t)| * (sum_{x in I(a_t)} MD(t)[x] + G_t),  G_parent += gamma_t
// The result is exactly Alg. 4's (up to FP32 rounding); the work is one pull per slot instead of
// q-1 pushes per tree node.  The score vectors of one depth form an [n] x pitch FP32 matrix in the ColLayout
// of internal.cuh: node-major up to 256 columns, else groups of 256 columns, each an [n][256] block.
#include <algorithm>

#include "internal.cuh"

namespace ps {

// zero columns [c0, c0 + w4 * 4) of every row (c0 a multiple of 4), one float4 per thread; consecutive
// threads take consecutive float4s of a row
__global__ void k_zero_cols(int32_t n, float *MD, ColLayout L, int32_t c0, int32_t w4) {
    const int64_t total = (int64_t)n * w4;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t v = i / w4;
        const int32_t c = c0 + 4 * (int32_t)(i - v * w4);
        *reinterpret_cast<float4 *>(MD + L.at(v, c)) = make_float4(0.f, 0.f, 0.f, 0.f);
    }
}

// zero columns [c0, c1) of every row, c1 - c0 < 4 (the head of a range that does not start on a float4)
__global__ void k_zero_cols_head(int32_t n, float *MD, ColLayout L, int32_t c0, int32_t c1) {
    const int64_t v = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (v >= n) return;
    for (int32_t c = c0; c < c1; ++c) MD[L.at(v, c)] = 0.f;
}

// zeroes columns [c0, c0 + width) rounded up to a multiple of 4 (inside the pitch)
void launch_zero_cols(int32_t n, float *MD, ColLayout L, int32_t c0, int32_t width, cudaStream_t s) {
    if (width <= 0) return;
    const int32_t end = (c0 + width + 3) / 4 * 4, a0 = (c0 + 3) / 4 * 4;
    if (a0 > c0) k_zero_cols_head<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, MD, L, c0, std::min(a0, end));
    if (end > a0) {
        const int32_t w4 = (end - a0) / 4;
        const int blocks = grid_for((int64_t)n * w4, 256, 8);
        k_zero_cols<<<blocks, 256, 0, s>>>(n, MD, L, a0, w4);
    }
}

// a tree node with a push column: subtree height 2, below the super-root
__device__ __forceinline__ bool is_push_node(const TrieTable &t, int32_t e) { return t.height[e] == 2 && t.depth[e] != 0; }

// ------------------------------------------------------------------------------------------------
// scatter: for every tree node g at depth t+2 whose grandparent is dense,
// D[a_g][slot(grandparent(g))] += gamma_g.
// ------------------------------------------------------------------------------------------------
// The same launch zeroes what the pull needs zeroed: the spare row n of B, which its padding gathers read, and in A the
// rows of vertices whose in-list is cut into several pieces, which receive atomic adds.  (Three launches a level were a
// sixth of a call on a graph of 1,000 nodes.)
__global__ void __launch_bounds__(256) k_prepare_pull(const int32_t *__restrict__ nodes, int32_t cnt, int32_t blocks_sc,
                                                      TrieTable t, float *B, ColLayout Lb,
                                                      const int32_t *__restrict__ rows, int32_t nrows, float *A,
                                                      ColLayout La, int32_t width, int32_t zrows, int32_t z0,
                                                      int32_t zw) {
    pdl_wait();
    if ((int32_t)blockIdx.x < blocks_sc) {
        const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
        if (i >= cnt) return;
        const int32_t e = nodes[i];
        const int32_t gp = t.parent[t.parent[e]];
        const int32_t sl = t.slot[gp];
        if (sl < 0 || is_push_node(t, gp)) return;
        atomicAdd(B + Lb.at(t.node[e], sl), t.gamma[e]);
        return;
    }
    const int64_t total = ((int64_t)nrows + 1) * width;
    const int64_t step = (int64_t)(gridDim.x - blocks_sc) * blockDim.x;
    for (int64_t i = (int64_t)(blockIdx.x - blocks_sc) * blockDim.x + threadIdx.x; i < total; i += step) {
        const int64_t r = i / width;
        const int32_t c = (int32_t)(i - r * width);
        if (r < nrows) A[La.at(rows[r], c)] = 0.f;
        else B[Lb.at(Lb.n, c)] = 0.f;
    }
    const int64_t block = (int64_t)zrows * zw;
    for (int64_t i = (int64_t)(blockIdx.x - blocks_sc) * blockDim.x + threadIdx.x; i < block; i += step) {
        const int64_t r = i / zw;
        A[La.at(r, z0 + (int32_t)(i - r * zw))] = 0.f;
    }
}

// nodes: the tree nodes two depths down (cnt may be 0); width: the columns pulled
void launch_prepare_pull(const DeviceGraph &g, const int32_t *nodes, int32_t cnt, TrieTable t, float *B, ColLayout Lb,
                         float *A, ColLayout La, int32_t width, int32_t zrows, int32_t z0, int32_t zw, cudaStream_t s) {
    const int bs = (std::max(0, cnt) + 255) / 256;
    const int bz = grid_for(std::max(((int64_t)g.n_split + 1) * std::max(1, width), (int64_t)zrows * zw), 256, 8);
    pdl_launch(k_prepare_pull, dim3(bs + bz), dim3(256), 0, s, nodes, cnt, bs, t, B, Lb, g.split_v, g.n_split, A, La, width,
               zrows, z0, zw);
}

// ------------------------------------------------------------------------------------------------
// push: for every tree node g at depth t+2 whose grandparent p is a push node:
// MD[x][slot(p)] += sqrt(c)/|I(x)| * gamma_g for every x in O(a_g).  A push node's column is either in the
// push block of its depth (slot >= h0) or the column it inherited from its parent (slot < h0); a launch
// serves one of the two kinds or both.  One block per node g: an out-list can hold tens of thousands of edges
// (hubs), so the block's threads split it and a hub does not hold up the launch.
// ------------------------------------------------------------------------------------------------
// A block per node waits for its longest list: few nodes get larger blocks, so a hub's list takes fewer rounds.
// (R-MAT 2^20, one query: 0.84 ms in 49 launches with 128 threads and one edge a round, 0.48 now.)
static int list_threads(int32_t cnt) {
    return cnt <= 1024 ? 512 : (cnt <= 4096 ? 256 : 128);
}

__global__ void __launch_bounds__(512) k_push_h2(const int64_t *__restrict__ out_off, const int32_t *__restrict__ out_col,
                                                 const float *__restrict__ w, const int32_t *__restrict__ nodes,
                                                 TrieTable t, float *MD, ColLayout L, int32_t h0, int32_t which,
                                                 int32_t rows) {
    pdl_wait();
    const int32_t e = nodes[blockIdx.x];
    const int32_t p = t.parent[t.parent[e]];  // the height-2 node
    const int32_t sl = t.slot[p];
    if (sl < 0 || !is_push_node(t, p) || (which != 2 && (sl < h0) != (which == 1))) return;
    const int32_t a = t.node[e];
    const float g = t.gamma[e];
    const int64_t beg = out_off[a], end = out_off[a + 1];
    float *col = MD + L.base(sl);
    const int32_t rp = L.rpitch(sl);
    for (int64_t k = beg + threadIdx.x; k < end; k += 4 * blockDim.x) {
        int32_t x[4];
        float wx[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            const int64_t ku = k + u * (int64_t)blockDim.x;
            x[u] = ku < end ? __ldg(out_col + ku) : rows;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) wx[u] = x[u] < rows ? __ldg(w + x[u]) : 0.f;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (x[u] < rows) atomicAdd(col + (int64_t)x[u] * rp, wx[u] * g);  // rows nobody reads are left out
    }
}

void launch_push_h2(const DeviceGraph &g, const int32_t *nodes, int32_t cnt, TrieTable t, float *MD, ColLayout L,
                    int32_t h0, int32_t which, cudaStream_t s) {
    if (cnt <= 0) return;
    pdl_launch(k_push_h2, dim3(cnt), dim3(list_threads(cnt)), 0, s, g.out_off, g.out_col, g.w, nodes, t, MD, L, h0, which,
               g.n_active);
}

// ------------------------------------------------------------------------------------------------
// accumulate: D of the dense nodes of a depth, in place in the previous level's MD buffer.  A dense node's
// column already holds its heir's MD (the heir inherits the column); each group g adds (or, for a node
// without heir, sets) the sum of its other children's columns: B[v][dst_g] (+)= sum of B[v][src], src in
// srcs[off_g .. off_g+1).  No destination is a source of any group (the column assignment guarantees it), so
// the groups are independent.  Groups are cut into parts of at most four sources; the first parts of all groups run
// before the others, which add atomically.  A lane holds a part -- its offsets in a row, computed once -- and its warp
// walks down the rows, four at a time, so 16 loads are in flight per lane and nothing but the scores is read per row.
// Later parts of one group sit in neighbouring lanes: they are summed by shuffles before one lane adds, since a node
// with thousands of children would queue thousands of adds on one address.
// Only rows below n_active are accumulated: a row of a node without out-edges is never read once accumulated (the
// pull and the gamma gather in-neighbours' rows), and the renumbering puts those nodes last.
// In place it serves depths with few sources (k_accumulate_rows the others).
// ------------------------------------------------------------------------------------------------
constexpr int kAccRows = 4;

template <bool LATER>
__global__ void __launch_bounds__(256) k_accumulate(int32_t n, float *B, ColLayout L, const int32_t *__restrict__ pdst,
                                                    const int4 *__restrict__ psrc, int32_t np) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int32_t pi = blockIdx.y * 32 + lane;
    const bool on = pi < np;
    const int32_t d = on ? __ldg(pdst + pi) : 0;
    const int4 sc = on ? __ldg(psrc + pi) : make_int4(-1, -1, -1, -1);
    const int32_t rp = L.rpitch(0);
    float *dst = B + L.base(d & 0x3fffffff);
    const float *s0 = B + L.base(max(sc.x, 0)), *s1 = B + L.base(max(sc.y, 0)), *s2 = B + L.base(max(sc.z, 0)),
                *s3 = B + L.base(max(sc.w, 0));
    const bool set = d & (1 << 30);  // no heir: the column is set
    // LATER: the lanes of one group are a run; its first lane adds the run's sum
    const int32_t key = on ? d : -1 - lane;
    const int32_t prev = __shfl_up_sync(0xffffffffu, key, 1);
    const bool head = lane == 0 || prev != key;
    const unsigned heads = __ballot_sync(0xffffffffu, head);
    const int run_end = lane == 31 ? 32 : ((heads >> (lane + 1)) ? lane + __ffs(heads >> (lane + 1)) : 32);
    const bool runs = LATER && heads != 0xffffffffu;
    const int64_t step = (int64_t)gridDim.x * (blockDim.x >> 5) * kAccRows;
    for (int64_t v0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * kAccRows; v0 < n; v0 += step) {
        float sum[kAccRows];
#pragma unroll
        for (int u = 0; u < kAccRows; ++u) {
            const int64_t o = min(v0 + u, (int64_t)n - 1) * rp;
            sum[u] = sc.x >= 0 ? s0[o] : 0.f;
            if (sc.y >= 0) sum[u] += s1[o];
            if (sc.z >= 0) sum[u] += s2[o];
            if (sc.w >= 0) sum[u] += s3[o];
        }
        if (runs) {
#pragma unroll
            for (int u = 0; u < kAccRows; ++u)
                for (int o = 1; o < 32; o <<= 1) {
                    const float y = __shfl_down_sync(0xffffffffu, sum[u], o);
                    if (lane + o < run_end) sum[u] += y;
                }
        }
#pragma unroll
        for (int u = 0; u < kAccRows; ++u) {
            if (!on || v0 + u >= n) continue;
            float *p = dst + (v0 + u) * rp;
            if (LATER) {
                if (head) atomicAdd(p, sum[u]);
            } else {
                *p = set ? sum[u] : *p + sum[u];
            }
        }
    }
}

// The same with whole rows staged: a block brings R rows (W columns each) into shared memory with asynchronous copies,
// forms every group's sum there and writes the destinations back.  A part's sources lie anywhere in a row, so in place
// each source costs a sector, and the parts of different warps fetch one sector several times over: with thousands of
// sources the in-place kernel read 58 GB for a 1.9 GB matrix.  Staged, a row is read once, in order.  R is as large as
// lets two blocks share an SM, so one block's copies run under the other's sums; part records are read once per R rows.
constexpr int kStageThreads = 512;
constexpr size_t kStageBytes = 224 * 1024;  // shared memory of the blocks on one SM

template <int R>
__global__ void __launch_bounds__(kStageThreads) k_accumulate_rows(int32_t n, float *B, ColLayout L, int32_t W,
                                                                   const int32_t *__restrict__ p1dst,
                                                                   const int4 *__restrict__ p1src, int32_t np1,
                                                                   const int32_t *__restrict__ p2dst,
                                                                   const int4 *__restrict__ p2src, int32_t np2) {
    extern __shared__ __align__(16) float rows[];
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const uint32_t rows_s = (uint32_t)__cvta_generic_to_shared(rows);
    auto part = [&](const float *row, int4 sc) {
        float s = sc.x >= 0 ? row[sc.x] : 0.f;
        if (sc.y >= 0) s += row[sc.y];
        if (sc.z >= 0) s += row[sc.z];
        if (sc.w >= 0) s += row[sc.w];
        return s;
    };
    for (int64_t v0 = (int64_t)blockIdx.x * R; v0 < n; v0 += (int64_t)gridDim.x * R) {
        const int nr = (int)min((int64_t)R, n - v0);
        for (int r = 0; r < nr; ++r)
            for (int32_t c = 4 * threadIdx.x; c < W; c += 4 * kStageThreads)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(rows_s + 4 * (r * W + c)),
                             "l"(B + L.at(v0 + r, c))
                             : "memory");
        asm volatile("cp.async.wait_all;" ::: "memory");
        __syncthreads();
        for (int32_t pi = threadIdx.x; pi < np1; pi += kStageThreads) {
            const int32_t d = __ldg(p1dst + pi), c = d & 0x3fffffff;
            const int4 sc = __ldg(p1src + pi);
            for (int r = 0; r < nr; ++r) {
                float *row = rows + r * W;
                const float s = part(row, sc);
                row[c] = (d & (1 << 30)) ? s : row[c] + s;  // bit 30: no heir, the column is set
            }
        }
        __syncthreads();
        if (np2 > 0) {
            for (int32_t p0 = threadIdx.x & ~31; p0 < np2; p0 += kStageThreads) {
                const int32_t pi = p0 + lane;
                const bool on = pi < np2;
                const int32_t d = on ? __ldg(p2dst + pi) : -1 - lane;
                const int4 sc = on ? __ldg(p2src + pi) : make_int4(-1, -1, -1, -1);
                const int32_t prev = __shfl_up_sync(0xffffffffu, d, 1);
                const bool head = lane == 0 || prev != d;
                const unsigned heads = __ballot_sync(0xffffffffu, head);
                const int run_end = lane == 31 || !(heads >> (lane + 1)) ? 32 : lane + __ffs(heads >> (lane + 1));
                for (int r = 0; r < nr; ++r) {
                    float s = part(rows + r * W, sc);
                    for (int o = 1; o < 32; o <<= 1) {
                        const float y = __shfl_down_sync(0xffffffffu, s, o);
                        if (lane + o < run_end) s += y;
                    }
                    if (on && head) atomicAdd(rows + r * W + d, s);
                }
            }
            __syncthreads();
        }
        for (int32_t pi = threadIdx.x; pi < np1; pi += kStageThreads) {
            const int32_t c = __ldg(p1dst + pi) & 0x3fffffff;
            for (int r = 0; r < nr; ++r) B[L.at(v0 + r, c)] = rows[r * W + c];
        }
        __syncthreads();
    }
}

template <int R>
static cudaError_t accumulate_rows(int32_t n, float *B, const ColLayout &L, int32_t W, const int32_t *p1dst,
                                   const int4 *p1src, int32_t np1, const int32_t *p2dst, const int4 *p2src, int32_t np2,
                                   cudaStream_t s) {
    const size_t bytes = (size_t)R * W * sizeof(float);
    // the same for every call: the attribute belongs to the kernel, and calls of other threads launch it with other sizes
    const cudaError_t e = cudaFuncSetAttribute(k_accumulate_rows<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                               (int)kStageBytes);
    if (e != cudaSuccess) return e;
    const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(4, kStageBytes / std::max<size_t>(1, bytes)));
    return pdl_launch(k_accumulate_rows<R>, dim3(grid_for(((int64_t)n + R - 1) / R, 1, per_sm)), dim3(kStageThreads), bytes,
                      s, n, B, L, W, p1dst, p1src, np1, p2dst, p2src, np2);
}

// W: the columns of a row that hold data; nsrc: the sources of all parts.  In place, a row costs a sector per source and
// destination, staged the whole row: rows are staged when the former would touch as many bytes.  Two eps = 0.05 queries on
// R-MAT 2^18: 11.2 ms in four launches with a warp per row in place, 13.3 with a lane per part in place, 3.1 staged by
// this rule; the headline query 1.7, 2.6 and 2.5 ms (its calls 20.4, 20.2 and 20.2 ms).
cudaError_t launch_accumulate(int32_t n, float *B, ColLayout L, int32_t W, int64_t nsrc, const int32_t *p1dst,
                              const int4 *p1src, int32_t np1, const int32_t *p2dst, const int4 *p2src, int32_t np2,
                              cudaStream_t s) {
    if (np1 <= 0 || n <= 0) return cudaSuccess;
    const size_t row = (size_t)W * sizeof(float);
    if (8 * (nsrc + np1) >= W && row <= kStageBytes) {
        if (8 * row <= kStageBytes / 2) return accumulate_rows<8>(n, B, L, W, p1dst, p1src, np1, p2dst, p2src, np2, s);
        if (4 * row <= kStageBytes / 2) return accumulate_rows<4>(n, B, L, W, p1dst, p1src, np1, p2dst, p2src, np2, s);
        if (2 * row <= kStageBytes / 2) return accumulate_rows<2>(n, B, L, W, p1dst, p1src, np1, p2dst, p2src, np2, s);
        return accumulate_rows<1>(n, B, L, W, p1dst, p1src, np1, p2dst, p2src, np2, s);
    }
    auto grid = [&](int32_t np) {
        const int y = (np + 31) / 32;
        const int x = grid_for((int64_t)(n + kAccRows - 1) / kAccRows * 32, 256, 8);
        return dim3((unsigned)std::max(1, std::min(x, 8 * 152 / y + 1)), (unsigned)y);
    };
    cudaError_t e = pdl_launch(k_accumulate<false>, grid(np1), dim3(256), 0, s, n, B, L, p1dst, p1src, np1);
    if (e == cudaSuccess && np2 > 0)
        e = pdl_launch(k_accumulate<true>, grid(np2), dim3(256), 0, s, n, B, L, p2dst, p2src, np2);
    return e;
}

// ------------------------------------------------------------------------------------------------
// gamma, for every tree node t at the current depth:
//   beta_t  = sqrt(c)/|I(a_t)| * (sum_{x in I(a_t)} MD(t)[x] + G_t)   (the score PROBE would give a_t)
//   gamma_t = w_t / n_r - beta_t;  G_parent += gamma_t
// ------------------------------------------------------------------------------------------------
// One block per tree node (the in-list of a hub is long; see list_threads); four independent gathers per thread in
// flight.  (R-MAT 2^20, one query: 1.06 ms in 40 launches with 128 threads, 0.63 now.)
__global__ void __launch_bounds__(512) k_gamma(const int64_t *__restrict__ in_off, const int32_t *__restrict__ in_col,
                                               const float *__restrict__ w, const int32_t *__restrict__ nodes,
                                               TrieTable t, const float *__restrict__ inv_nr,
                                               const float *MD, ColLayout Lc) {
    __shared__ float part[16];
    pdl_wait();
    const int32_t e = nodes[blockIdx.x];
    const int32_t a = t.node[e];
    const int32_t sl = t.slot[e];
    float sum = 0.f;
    if (sl >= 0 && MD != nullptr) {
        const int64_t beg = in_off[a], end = in_off[a + 1];
        const float *col = MD + Lc.base(sl);
        const int32_t rp = Lc.rpitch(sl), T = blockDim.x;
        float s1 = 0.f, s2 = 0.f, s3 = 0.f;
        int64_t k = beg + threadIdx.x;
        for (; k + 3 * T < end; k += 4 * T) {
            const int32_t x0 = __ldg(in_col + k), x1 = __ldg(in_col + k + T);
            const int32_t x2 = __ldg(in_col + k + 2 * T), x3 = __ldg(in_col + k + 3 * T);
            sum += col[(int64_t)x0 * rp];
            s1 += col[(int64_t)x1 * rp];
            s2 += col[(int64_t)x2 * rp];
            s3 += col[(int64_t)x3 * rp];
        }
        for (; k < end; k += T) sum += col[(int64_t)__ldg(in_col + k) * rp];
        sum += s1 + s2 + s3;
    }
    for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x == 0) {
        float tot = 0.f;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += part[i];
        const float beta = __ldg(w + a) * (tot + t.G[e]);
        const float g = (float)t.weight[e] * inv_nr[t.query[e]] - beta;
        t.gamma[e] = g;
        const int32_t p = t.parent[e];
        if (p >= 0) atomicAdd(&t.G[p], g);
    }
}

void launch_gamma(const DeviceGraph &g, const int32_t *nodes, int32_t cnt, TrieTable t, const float *inv_nr,
                  const float *MD, ColLayout L, cudaStream_t s) {
    if (cnt <= 0) return;
    pdl_launch(k_gamma, dim3(cnt), dim3(list_threads(cnt)), 0, s, g.in_off, g.in_col, g.w, nodes, t, inv_nr, MD, L);
}

// ------------------------------------------------------------------------------------------------
// finalize: out[q][v] = MD0[ext2int[v]][rho_slot(q)] + shift for the caller's node id v, out[q][u_q] = 1 (s(u,u) = 1).
// ------------------------------------------------------------------------------------------------
__global__ void k_finalize(int32_t n, int32_t B, const int32_t *__restrict__ qnode, const int32_t *__restrict__ rho_slot,
                           const float *__restrict__ MD0, ColLayout L, const int32_t *__restrict__ ext2int,
                           float shift, float *__restrict__ out) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    const int32_t q = blockIdx.y;
    if (i >= n) return;
    const int32_t sl = rho_slot[q];
    float v = (sl >= 0 ? MD0[L.at(ext2int[i], sl)] : 0.f) + shift;
    if ((int32_t)i == qnode[q]) v = 1.f;
    out[(int64_t)q * n + i] = v;
}

void launch_finalize(int32_t n, int32_t B, const int32_t *qnode, const int32_t *rho_slot, const float *MD0,
                     ColLayout L, const int32_t *ext2int, float shift, float *out, cudaStream_t s) {
    dim3 grid((unsigned)((n + 255) / 256), (unsigned)B);
    k_finalize<<<grid, 256, 0, s>>>(n, B, qnode, rho_slot, MD0, L, ext2int, shift, out);
}

__global__ void k_map_ids(int32_t *ids, int64_t count, const int32_t *__restrict__ map) {
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < count && ids[i] >= 0) ids[i] = map[ids[i]];
}

void launch_map_ids(int32_t *ids, int64_t count, const int32_t *map, cudaStream_t s) {
    if (count <= 0) return;
    k_map_ids<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(ids, count, map);
}

}  // namespace ps
