// C ABI of libprobesim.so: the graph store, the query engine and the entry points of include/probesim.h.
#include <cuda_runtime.h>

#include <algorithm>
#include <chrono>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <vector>

#include "engine.cuh"

using namespace ps;

// ------------------------------------------------------------------------------------------------
// errors
// ------------------------------------------------------------------------------------------------
static thread_local std::string g_last_error;

void ps::set_last_error(const char *msg) { g_last_error = msg; }

static probesim_status fail(probesim_status st, const std::string &msg) {
    g_last_error = msg;
    return st;
}

probesim_status ps::fail_status(probesim_status st, const std::string &msg) { return fail(st, msg); }

#define PS_CUDA(expr)                                                                                  \
    do {                                                                                               \
        cudaError_t _e = (expr);                                                                       \
        if (_e != cudaSuccess) {                                                                       \
            return fail(_e == cudaErrorMemoryAllocation ? PROBESIM_E_NOMEM : PROBESIM_E_CUDA,          \
                        std::string(#expr) + ": " + cudaGetErrorString(_e));                           \
        }                                                                                              \
    } while (0)

// an allocation of one walk range's buffers in the randomized PROBE: when it fails, the range is split
#define PS_ALLOC_RANGE(expr)                                                                           \
    do {                                                                                               \
        cudaError_t _e = (expr);                                                                       \
        if (_e != cudaSuccess) {                                                                       \
            cudaGetLastError();                                                                        \
            *too_big = true;                                                                           \
            return fail(PROBESIM_E_NOMEM, std::string(#expr) + ": " + cudaGetErrorString(_e));         \
        }                                                                                              \
    } while (0)

// an allocation of a batch's working buffers: when it fails on a call of several queries, the caller splits it
#define PS_ALLOC(expr)                                                                                 \
    do {                                                                                               \
        cudaError_t _e = (expr);                                                                       \
        if (_e != cudaSuccess) {                                                                       \
            cudaGetLastError();                                                                        \
            *too_big = B > 1;                                                                          \
            return fail(PROBESIM_E_NOMEM, std::string(#expr) + ": " + cudaGetErrorString(_e));         \
        }                                                                                              \
    } while (0)

#define PS_TRY(expr)                                  \
    do {                                              \
        probesim_status _s = (expr);                  \
        if (_s != PROBESIM_OK) return _s;             \
    } while (0)

static uint32_t threshold_stop(double c) { return (uint32_t)std::floor((1.0 - std::sqrt(c)) * 4294967296.0); }
static uint32_t threshold_keep(double c) {
    const double t = std::floor(std::sqrt(c) * 4294967296.0);
    return t >= 4294967295.0 ? 4294967295u : (uint32_t)t;
}

static int64_t num_walks(double c, double eps, double delta, int64_t n) {
    return (int64_t)std::ceil(3.0 * c / (eps * eps) * std::log((double)n / delta));
}

int64_t ps::num_walks_for(const probesim_graph *g, double eps) { return num_walks(g->cfg.c, eps, g->cfg.delta, g->n); }

static bool is_device_ptr(const void *p) {
    if (!p) return false;
    cudaPointerAttributes a;
    cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

// host memory the CUDA runtime does not know: no copy or kernel in flight can still be writing it
static bool is_plain_host_ptr(const void *p) {
    cudaPointerAttributes a;
    const cudaError_t e = cudaPointerGetAttributes(&a, p);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeUnregistered;
}

// ------------------------------------------------------------------------------------------------
// graph store
// ------------------------------------------------------------------------------------------------

// Builds the device graph store from the caller's edge list (device arrays of the caller's ids) with the kernels
// of graph_build.cu and publishes it as the first version.  Repeated edges and loops are dropped.  Internally nodes
// are renumbered by descending out-degree (ties by the caller's id): the pull kernel gathers score rows of
// in-neighbours, which are mostly high-out-degree nodes, so their rows become contiguous and stay cached.  I(v)
// keeps the caller's source-id order (walks pick the k-th entry of that order) but holds internal ids; O(x) holds
// internal ids in ascending order; ext2int / int2ext map at the boundary.
static probesim_status build_graph(probesim_graph *g, int32_t n, const int32_t *d_src, const int32_t *d_dst, int64_t m,
                                   cudaStream_t st) {
    struct Scratch {  // the build's temporaries: parts of one allocation, freed on every return
        DevBuf slab;
        DevBuf ka, kb, kc, cnt, off, part, ext_off, outdeg, rka, rkb, indeg_i, outdeg_i, hist, flag;
        ~Scratch() { slab.release(); }
    } t;
    // parts of 256-byte multiples out of one allocation (an allocation and its release cost the host some 70 us)
    auto carve = [](DevBuf &slab, const std::vector<std::pair<DevBuf *, size_t>> &parts) -> cudaError_t {
        size_t total = 0;
        for (auto &x : parts) total += (x.second + 255) / 256 * 256;
        const cudaError_t e = slab.ensure_exact(total);
        if (e != cudaSuccess) return e;
        char *at = slab.as<char>();
        for (auto &x : parts) {
            x.first->set_view(at, x.second);
            at += (x.second + 255) / 256 * 256;
        }
        return cudaSuccess;
    };
    auto bitlen = [](uint64_t x) { int b = 0; while (x) { ++b; x >>= 1; } return b; };
    const int bs = std::max(1, bitlen((uint64_t)std::max(1, n - 1)));  // bits of a node id
    const uint32_t smask = (uint32_t)(((uint64_t)1 << bs) - 1);
    const uint64_t end_key = ((uint64_t)1 << 2 * bs) - 1;
    const int64_t M = std::max<int64_t>(1, m);
    const int64_t big = std::max<int64_t>(M, n);
    const int64_t ntiles = radix_tiles(big);
    const int nb = 2 * (kPiece + 1);  // piece buckets: rows with out-edges, then the others, by length
    const size_t n8 = 8 * (size_t)n;
    PS_CUDA(carve(t.slab, {{&t.ka, 8 * (size_t)(M + 1)}, {&t.kb, 8 * (size_t)(M + 1)}, {&t.kc, 8 * (size_t)M},
                           {&t.cnt, 8 * (size_t)(256 * ntiles)}, {&t.off, 8 * (size_t)(256 * ntiles + 1)},
                           {&t.part, 8 * (size_t)scan64_partials_needed(std::max<int64_t>(256 * ntiles, big + 1))},
                           {&t.flag, sizeof(int32_t)}, {&t.ext_off, n8 + 8}, {&t.outdeg, n8}, {&t.rka, n8}, {&t.rkb, n8},
                           {&t.indeg_i, n8}, {&t.outdeg_i, n8},
                           {&t.hist, sizeof(unsigned long long) * (2 * (size_t)nb + 2)}}));
    long long *cnt = t.cnt.as<long long>(), *off = t.off.as<long long>(), *part = t.part.as<long long>();
    // 1-3: sorted unique edge keys (dst << bs | src, caller's ids)
    PS_CUDA(cudaMemsetAsync(t.flag.p, 0, sizeof(int32_t), st));
    launch_build_keys(d_src, d_dst, m, n, bs, t.ka.as<uint64_t>(), t.flag.as<int32_t>(), st);
    int32_t bad = 0;
    PS_CUDA(cudaMemcpyAsync(&bad, t.flag.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    if (bad) return fail(PROBESIM_E_RANGE, "edge id outside [0, n)");
    uint64_t *sorted = radix_sort_u64(t.ka.as<uint64_t>(), t.kb.as<uint64_t>(), m, 0, 2 * bs, cnt, off, part, st);
    long long *pre = reinterpret_cast<long long *>(sorted == t.ka.as<uint64_t>() ? t.kb.p : t.ka.p);
    launch_build_flags(sorted, m, end_key, pre, st);
    launch_scan64(pre, m, part, pre, st);  // in place: pre[m] = the number of distinct edges
    long long mu_ll = 0;
    PS_CUDA(cudaMemcpyAsync(&mu_ll, pre + std::max<int64_t>(0, m), sizeof(long long), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    const int64_t mu = m > 0 ? (int64_t)mu_ll : 0;
    uint64_t *ukeys = t.kc.as<uint64_t>();
    launch_build_compact(sorted, m, end_key, pre, ukeys, st);
    // 4: in-list offsets and out-degrees by caller id, then the renumbering
    long long *ext_off = t.ext_off.as<long long>();
    unsigned long long *outdeg = t.outdeg.as<unsigned long long>();
    PS_CUDA(cudaMemsetAsync(outdeg, 0, 8 * (size_t)n, st));
    launch_build_ext_off(ukeys, mu, n, bs, ext_off, st);
    launch_build_outdeg(ukeys, mu, smask, outdeg, st);
    launch_build_rank_keys(outdeg, n, mu, bs, t.rka.as<uint64_t>(), st);
    const uint64_t *rk =
        radix_sort_u64(t.rka.as<uint64_t>(), t.rkb.as<uint64_t>(), n, bs, bs + bitlen((uint64_t)mu), cnt, off, part, st);
    PS_CUDA(g->ext2int.ensure(sizeof(int32_t) * n));
    PS_CUDA(g->int2ext.ensure(sizeof(int32_t) * n));
    launch_build_perm(rk, n, smask, ext_off, outdeg, g->int2ext.as<int32_t>(), g->ext2int.as<int32_t>(),
                      t.indeg_i.as<long long>(), t.outdeg_i.as<long long>(), st);
    // 5: the CSR arrays in internal ids
    auto sv = std::make_shared<StoreVersion>();
    const int64_t cap_pieces = (int64_t)n + mu / kPiece + 1;
    const size_t off_bytes = sizeof(int64_t) * ((size_t)n + 1), col_bytes = sizeof(int32_t) * std::max<int64_t>(1, mu);
    PS_CUDA(carve(sv->arena, {{&sv->in_off, off_bytes}, {&sv->out_off, off_bytes}, {&sv->in_col, col_bytes},
                              {&sv->out_col, col_bytes}, {&sv->w, sizeof(float) * (size_t)n},
                              {&sv->rec, sizeof(int4) * (size_t)n}, {&sv->piece_v, sizeof(int32_t) * (size_t)cap_pieces},
                              {&sv->piece_beg, sizeof(int64_t) * (size_t)cap_pieces},
                              {&sv->piece_len, sizeof(int32_t) * (size_t)cap_pieces},
                              {&sv->split_v, sizeof(int32_t) * (size_t)n}}));
    launch_scan64(t.indeg_i.as<long long>(), n, part, sv->in_off.as<long long>(), st);
    launch_scan64(t.outdeg_i.as<long long>(), n, part, sv->out_off.as<long long>(), st);
    uint64_t *okeys = t.ka.as<uint64_t>();  // the edge-key buffers are free again (the unique keys live in kc)
    launch_build_in_col(n, g->int2ext.as<int32_t>(), ext_off, sv->in_off.as<int64_t>(), ukeys, smask,
                        g->ext2int.as<int32_t>(), bs, sv->in_col.as<int32_t>(), okeys, st);
    const uint64_t *osorted = radix_sort_u64(okeys, t.kb.as<uint64_t>(), mu, bs, 2 * bs, cnt, off, part, st);
    launch_build_out_col(osorted, mu, smask, sv->out_col.as<int32_t>(), st);
    // w and the pull pieces (in-lists cut into at most kPiece edges, longest first)
    launch_upd_w(n, sv->in_off.as<long long>(), sv->in_col.as<int32_t>(), (float)std::sqrt(g->cfg.c),
                 g->int2ext.as<int32_t>(), rec_shift_for(n), sv->w.as<float>(), sv->rec.as<int4>(),
                 t.indeg_i.as<long long>(), st);
    unsigned long long *hist = t.hist.as<unsigned long long>(), *cursor = hist + nb, *nsplit = cursor + nb;
    PS_CUDA(cudaMemsetAsync(t.flag.p, 0, sizeof(int32_t), st));
    launch_active_rows(sv->out_off.as<int64_t>(), n, t.flag.as<int32_t>(), st);
    launch_upd_pieces(n, sv->in_off.as<long long>(), t.flag.as<int32_t>(), hist, cursor, sv->split_v.as<int32_t>(),
                      nsplit, sv->piece_v.as<int32_t>(), sv->piece_beg.as<int64_t>(), sv->piece_len.as<int32_t>(), st);
    std::vector<unsigned long long> hh(nb + 1);
    long long ends[2] = {0, 0};
    int32_t n_active = 0;
    PS_CUDA(cudaMemcpyAsync(&n_active, t.flag.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(hh.data(), hist, sizeof(unsigned long long) * nb, cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(hh.data() + nb, nsplit, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(&ends[0], sv->in_off.as<int64_t>() + n, 8, cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(&ends[1], sv->out_off.as<int64_t>() + n, 8, cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaGetLastError());
    PS_CUDA(cudaStreamSynchronize(st));
    if (ends[0] != mu || ends[1] != mu) return fail(PROBESIM_E_CUDA, "internal: the built lists disagree on m");
    int64_t npieces = 0, npieces_active = 0, m_active = 0;
    for (int k = 0; k < nb; ++k) {
        npieces += (int64_t)hh[k];
        if (k <= kPiece) npieces_active += (int64_t)hh[k], m_active += k * (int64_t)hh[k];  // bucket k: pieces of k edges
    }
    DeviceGraph &d = sv->dg;
    d.n = n;
    d.m = mu;
    d.in_off = sv->in_off.as<int64_t>();
    d.in_col = sv->in_col.as<int32_t>();
    d.out_off = sv->out_off.as<int64_t>();
    d.out_col = sv->out_col.as<int32_t>();
    d.w = sv->w.as<float>();
    d.rec = sv->rec.as<int4>();
    d.rec_shift = rec_shift_for(n);
    d.n_pieces = npieces;
    d.n_pieces_active = npieces_active;
    d.m_active = m_active;
    d.piece_v = sv->piece_v.as<int32_t>();
    d.piece_beg = sv->piece_beg.as<int64_t>();
    d.piece_len = sv->piece_len.as<int32_t>();
    d.n_split = (int32_t)hh[nb];
    d.n_active = n_active;
    d.split_v = sv->split_v.as<int32_t>();
    d.ext2int = g->ext2int.as<int32_t>();
    d.int2ext = g->int2ext.as<int32_t>();
    g->n = n;
    g->publish(sv);
    return PROBESIM_OK;
}

// Device memory one call on workspace ws may take (a server gives each worker a share of the graph's budget).
static size_t budget_of(const probesim_graph *g, const Workspace *ws) {
    return ws->budget ? ws->budget : g->budget.load();
}

// ------------------------------------------------------------------------------------------------
// query engine
// ------------------------------------------------------------------------------------------------
struct BatchPlan {
    int32_t B = 0, W = 0;
    std::vector<int32_t> node, base, k0;
    std::vector<uint32_t> qid;
    std::vector<float> inv_nr;
};

static probesim_status plan_batch(probesim_graph *g, const probesim_query *q, int32_t B, BatchPlan &P) {
    P.B = B;
    P.node.resize(B);
    P.base.resize(B + 1);
    P.k0.resize(B);
    P.qid.resize(B);
    P.inv_nr.resize(B);
    int64_t W = 0;
    for (int32_t b = 0; b < B; ++b) {
        const int64_t nr = num_walks(g->cfg.c, q[b].eps, g->cfg.delta, g->n);
        const int64_t kb = std::max<int64_t>(0, q[b].walk_begin);
        const int64_t ke = q[b].walk_end <= 0 ? nr : std::min<int64_t>(q[b].walk_end, nr);
        P.node[b] = q[b].node;
        P.qid[b] = q[b].query_id;
        P.k0[b] = (int32_t)std::min(kb, ke);
        P.base[b] = (int32_t)W;
        W += std::max<int64_t>(0, ke - kb);
        P.inv_nr[b] = (float)(1.0 / (double)nr);
        if (W > (int64_t)1 << 30) return fail(PROBESIM_E_INVALID, "too many walks in one call");
    }
    P.base[B] = (int32_t)W;
    P.W = (int32_t)W;
    return PROBESIM_OK;
}

// Uploads the batch arrays; returns the device view.
static probesim_status upload_batch(Workspace *ws, const BatchPlan &P, QueryBatch &qb, cudaStream_t st) {
    const int32_t B = P.B;
    const size_t bytes = sizeof(int32_t) * (4 * (size_t)B + 1) + sizeof(float) * B + 64;
    PS_CUDA(ws->pin_q.ensure(bytes));
    PS_CUDA(ws->qbuf.ensure(bytes));
    char *h = ws->pin_q.as<char>();
    int32_t *hn = reinterpret_cast<int32_t *>(h);
    std::memcpy(hn, P.node.data(), sizeof(int32_t) * B);
    std::memcpy(hn + B, P.qid.data(), sizeof(uint32_t) * B);
    std::memcpy(hn + 2 * B, P.base.data(), sizeof(int32_t) * (B + 1));
    std::memcpy(hn + 3 * B + 1, P.k0.data(), sizeof(int32_t) * B);
    std::memcpy(hn + 4 * B + 1, P.inv_nr.data(), sizeof(float) * B);
    PS_CUDA(cudaMemcpyAsync(ws->qbuf.p, h, bytes, cudaMemcpyHostToDevice, st));
    int32_t *d = ws->qbuf.as<int32_t>();
    qb.B = B;
    qb.node = d;
    qb.qid = reinterpret_cast<const uint32_t *>(d + B);
    qb.walk_base = d + 2 * B;
    qb.walk_k0 = d + 3 * B + 1;
    qb.inv_nr = reinterpret_cast<const float *>(d + 4 * B + 1);
    return PROBESIM_OK;
}

static int64_t next_pow2(int64_t x) {
    int64_t p = 1;
    while (p < x) p <<= 1;
    return p;
}

struct Timer {
    Workspace *ws;
    cudaStream_t st;
    size_t used = 0;
    cudaEvent_t get() {
        if (used == ws->ev.size()) {
            cudaEvent_t e;
            cudaEventCreate(&e);
            ws->ev.push_back(e);
        }
        return ws->ev[used++];
    }
};

// Brackets groups of launches with events when profiling is on; times are summed per phase after the
// batch's final synchronisation.
struct PhaseTimer {
    Timer *tm;
    bool on;
    std::vector<std::pair<int, std::pair<cudaEvent_t, cudaEvent_t>>> marks;
    int cur = -1;
    cudaEvent_t e0 = nullptr;
    void begin(int phase) {
        if (!on) return;
        cur = phase;
        e0 = tm->get();
        cudaEventRecord(e0, tm->st);
    }
    void end() {
        if (!on || cur < 0) return;
        cudaEvent_t e1 = tm->get();
        cudaEventRecord(e1, tm->st);
        marks.push_back({cur, {e0, e1}});
        cur = -1;
    }
    void collect(probesim_stats &st) {
        for (auto &m : marks) {
            float ms = 0.f;
            if (cudaEventElapsedTime(&ms, m.second.first, m.second.second) == cudaSuccess) st.phase_ms[m.first] += ms;
        }
    }
};

// The pull of a depth's nfull full 32-column tiles, from column 0 of B and A, in the tuning's shape (pull_shape.h); the
// level loop and the tuner launch it.  err: the TMA shape's error flag.
static cudaError_t pull_full(const DeviceGraph &g, const PullTuning &t, const float *B, const ColLayout &Lb, float *A,
                             const ColLayout &La, int32_t nfull, const uint32_t *zmask, int32_t *err, int64_t *launches,
                             cudaStream_t st) {
    if (nfull <= 0) return cudaSuccess;
    if (t.shape == kPullTma) {
        ++*launches;
        return launch_pull_tma(g, B, Lb.rpitch(0), Lb.K > 0 ? kGroup : Lb.R, Lb.tile_stride(), Lb.tile_sub(32), A,
                               La.rpitch(0), La.tile_stride(), La.tile_sub(32), nfull, t.bps[kPullTma], zmask, err, st);
    }
    const int32_t tw = t.shape == 16 ? 16 : 32;
    FullTiles f{32, 1, 0, nfull};
    if (t.shape == 32) f = full_tiles(nfull, g.n_pieces, g.n_active);
    if (f.wide > 0) {
        launch_pull(g, B, Lb.rpitch(0), Lb.tile_stride(), Lb.tile_sub(32 * f.per), A, La.rpitch(0), La.tile_stride(),
                    La.tile_sub(32 * f.per), f.wide, f.tile, t.bps[f.tile], zmask, st);
        ++*launches;
    }
    // all of the launch's tiles, or up to three that lie in one group after the wide ones
    const int32_t c0 = 32 * f.per * f.wide, one = 1 << 30;
    if (f.rest > 0) {
        launch_pull(g, B + Lb.base(c0), Lb.rpitch(0), Lb.tile_stride(), f.wide > 0 ? one : Lb.tile_sub(tw),
                    A + La.base(c0), La.rpitch(0), La.tile_stride(), f.wide > 0 ? one : La.tile_sub(tw),
                    f.rest * (32 / tw), t.shape, t.bps[t.shape], zmask ? zmask + c0 / 32 : nullptr, st);
        ++*launches;
    }
    return cudaSuccess;
}

// The pull of a tail tile of `tail` columns that starts at column c (it lies inside one group, or row, of each layout).
static void pull_tail(const DeviceGraph &g, const PullTuning &t, const float *B, const ColLayout &Lb, float *A,
                      const ColLayout &La, int32_t c, int32_t tail, const uint32_t *zmask, cudaStream_t st) {
    if (narrow_tail(g.n_pieces))
        launch_pull_narrow(g, B + Lb.base(c), Lb.rpitch(c), A + La.base(c), La.rpitch(c), tail, t.narrow[tail], zmask, st);
    else
        launch_pull(g, B + Lb.base(c), Lb.rpitch(c), 0, 1 << 30, A + La.base(c), La.rpitch(c), 0, 1 << 30, 1, tail,
                    t.bps[tail], zmask, st);
}

// Runs the query path for one batch into d_out ([B][n] on the device).  Returns PROBESIM_E_NOMEM with
// *too_big set when the level buffers of this batch would exceed the workspace budget.
static probesim_status run_batch(probesim_graph *g, Workspace *ws, const probesim_query *q, int32_t B, float *d_out,
                                 cudaStream_t st, bool *too_big) {
    *too_big = false;
    const DeviceGraph &dg = ws->dg;
    const int32_t n = dg.n;
    const int32_t L = g->cfg.l_max;
    BatchPlan P;
    PS_TRY(plan_batch(g, q, B, P));
    if ((size_t)P.W * L * 4 > budget_of(g, ws) / 4 && B > 1) {
        *too_big = true;
        return PROBESIM_E_NOMEM;
    }
    QueryBatch qb;
    PS_TRY(upload_batch(ws, P, qb, st));
    int64_t launches = 0;
    Timer tm{ws, st};
    PhaseTimer ph{&tm, ws->profiling != 0};
    // 1. walks (Def. 3)
    PS_CUDA(ws->walks.ensure(sizeof(int32_t) * std::max<int64_t>(1, (int64_t)P.W * L)));
    PS_CUDA(ws->lens.ensure(sizeof(int32_t) * std::max<int32_t>(1, P.W)));
    PS_CUDA(ws->ctr.ensure(sizeof(LaunchCounters)));
    LaunchCounters *d_ctr = ws->ctr.as<LaunchCounters>();
    PS_CUDA(cudaMemsetAsync(d_ctr, 0, sizeof(LaunchCounters), st));
    ph.begin(0);
    launch_walks(dg, qb, P.W, L, g->t_stop, g->cfg.seed, ws->walks.as<int32_t>(), ws->lens.as<int32_t>(), false, d_ctr, st);
    ph.end();
    ++launches;
    LaunchCounters *h_ctr = ws->pin_s.as<LaunchCounters>();
    PS_CUDA(cudaMemcpyAsync(h_ctr, d_ctr, sizeof(LaunchCounters), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    const int64_t walk_nodes = (int64_t)h_ctr->walk_nodes;
    ws->stats.walks += P.W;
    ws->stats.walk_nodes += walk_nodes;
    // 2. reverse-reachability tree (Alg. 4) in a hash table at load <= 1/2
    TrieTable t;
    t.cap = next_pow2(std::max<int64_t>(1024, 2 * (walk_nodes + B) + 64));
    const size_t cap = (size_t)t.cap;
    PS_CUDA(ws->t_key.ensure(8 * cap));
    PS_CUDA(ws->t_node.ensure(4 * cap));
    PS_CUDA(ws->t_parent.ensure(4 * cap));
    PS_CUDA(ws->t_depth.ensure(4 * cap));
    PS_CUDA(ws->t_query.ensure(4 * cap));
    PS_CUDA(ws->t_weight.ensure(4 * cap));
    PS_CUDA(ws->t_height.ensure(4 * cap));
    PS_CUDA(ws->t_slot.ensure(4 * cap));
    PS_CUDA(ws->t_gamma.ensure(4 * cap));
    PS_CUDA(ws->t_G.ensure(4 * cap));
    t.key = ws->t_key.as<unsigned long long>();
    t.node = ws->t_node.as<int32_t>();
    t.parent = ws->t_parent.as<int32_t>();
    t.depth = ws->t_depth.as<int32_t>();
    t.query = ws->t_query.as<int32_t>();
    t.weight = ws->t_weight.as<int32_t>();
    t.height = ws->t_height.as<int32_t>();
    t.slot = ws->t_slot.as<int32_t>();
    t.gamma = ws->t_gamma.as<float>();
    t.G = ws->t_G.as<float>();
    ph.begin(1);
    PS_CUDA(cudaMemsetAsync(t.key, 0xFF, 8 * cap, st));
    PS_CUDA(cudaMemsetAsync(t.weight, 0, 4 * cap, st));
    PS_CUDA(cudaMemsetAsync(t.height, 0, 4 * cap, st));
    PS_CUDA(cudaMemsetAsync(t.G, 0, 4 * cap, st));
    launch_trie_insert(dg, qb, P.W, L, ws->walks.as<int32_t>(), ws->lens.as<int32_t>(), t, d_ctr, st);
    ++launches;
    // 3. level schedule: the tree's nodes per depth, and the nodes that own a column (exported to pinned memory).  Every
    // dense node's heir takes over its column one depth down, so along a chain of heirs the MD column of the child
    // already is the D column of the parent and nothing is copied.  Push columns (height 2) sit in a block after the
    // dense columns.
    const int32_t D1 = L + 2;
    const int64_t most = walk_nodes + B;  // tree nodes
    PS_CUDA(ws->counts.ensure(sizeof(int32_t) * (4 * D1 + 1)));
    PS_CUDA(ws->node_list.ensure(sizeof(int32_t) * most));
    PS_CUDA(ws->pin_q.ensure(sizeof(int32_t) * 3 * (size_t)most));
    int32_t *d_count = ws->counts.as<int32_t>();
    const int32_t *h_exp = ws->pin_q.as<int32_t>();
    PS_CUDA(cudaMemsetAsync(d_count, 0, sizeof(int32_t) * (4 * D1 + 1), st));
    launch_sched(t, D1, d_count, d_count + 3 * D1, ws->node_list.as<int32_t>(), ws->pin_q.as<int32_t>(), most, st);
    ph.end();
    launches += 2;
    int32_t *h_cnt = reinterpret_cast<int32_t *>(ws->pin_s.as<char>() + 256);
    PS_CUDA(cudaMemcpyAsync(h_cnt, d_count, sizeof(int32_t) * 3 * D1, cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(h_ctr, d_ctr, sizeof(LaunchCounters), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    if (h_ctr->overflow) return fail(PROBESIM_E_CUDA, "internal: walk tree table overflow");
    const auto host0 = std::chrono::steady_clock::now();  // the host-side schedule starts (the device waits)
    std::vector<int32_t> ncount(D1), node_off(D1 + 1, 0);
    const int32_t *scount = h_cnt + D1, *hcount = h_cnt + 2 * D1;
    int32_t Dmax = 0, ncol_nodes = 0;
    for (int32_t d = 0; d < D1; ++d) {
        ncount[d] = h_cnt[d] + scount[d] + hcount[d];
        node_off[d + 1] = node_off[d] + ncount[d];
        ncol_nodes += scount[d] + hcount[d];
        if (ncount[d] > 0) Dmax = d;
    }
    ws->stats.tree_nodes += node_off[D1];
    ws->stats.vectors += ncol_nodes;
    LevelPlan &plan = ws->plan;
    if (!plan.build(ncol_nodes, h_exp, h_exp + most, h_exp + 2 * most, t.cap, B, D1,
                    [](int32_t rem) { return pull_tile_for(rem, 16); }))
        return fail(PROBESIM_E_CUDA, "internal: a tree node without its parent");
    const std::vector<int32_t> &nfull = plan.nfull, &tail = plan.tail, &dw = plan.dw, &hinh = plan.hinh, &h0v = plan.h0,
                               &rpv = plan.cols, &zoff = plan.zoff, &zany = plan.zany, &p1_at = plan.p1_at,
                               &p2_at = plan.p2_at;
    const std::vector<int64_t> &acc_src = plan.acc_src;
    std::vector<ColLayout> lay(D1);
    int64_t max_floats = 4 * (int64_t)n;
    for (int32_t d = 0; d <= Dmax; ++d) {
        lay[d] = make_layout(n, rpv[d]);
        max_floats = std::max<int64_t>(max_floats, lay[d].size());
        ws->stats.max_columns = std::max<int64_t>(ws->stats.max_columns, rpv[d]);
    }
    const size_t level_bytes2 = 2 * (size_t)max_floats * sizeof(float);
    if (level_bytes2 > budget_of(g, ws)) {
        *too_big = B > 1;
        return fail(PROBESIM_E_NOMEM, "score vectors of one query exceed the workspace budget");
    }
    // upload: entries and their columns, super-root columns, part destinations, zero masks, part sources (int4, 16-byte
    // aligned)
    const size_t sched_ints = 2 * (size_t)ncol_nodes + B + plan.p1dst.size() + plan.p2dst.size() + plan.zmask.size() +
                              plan.p1src.size() + plan.p2src.size() + 8;
    PS_CUDA(ws->sched.ensure(sizeof(int32_t) * sched_ints));
    PS_CUDA(ws->pin_q.ensure(sizeof(int32_t) * sched_ints));
    int32_t *h_sched = ws->pin_q.as<int32_t>();
    size_t o = 0;
    auto put = [&](const std::vector<int32_t> &v) {
        const size_t at = o;
        if (!v.empty()) std::memcpy(h_sched + o, v.data(), sizeof(int32_t) * v.size());
        o += v.size();
        return at;
    };
    const size_t o_ent = put(plan.ent), o_col = put(plan.col), o_rho = put(plan.rho), o_p1dst = put(plan.p1dst),
                 o_p2dst = put(plan.p2dst), o_zmask = put(plan.zmask);
    o = (o + 3) / 4 * 4;
    const size_t o_p1src = put(plan.p1src), o_p2src = put(plan.p2src);
    int32_t *d_sched = ws->sched.as<int32_t>();
    PS_CUDA(cudaMemcpyAsync(d_sched, h_sched, sizeof(int32_t) * o, cudaMemcpyHostToDevice, st));
    ws->stats.phase_ms[9] += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - host0).count();
    launch_set_slots(t, d_sched + o_ent, d_sched + o_col, ncol_nodes, st);
    ++launches;
    const int32_t *d_rho = d_sched + o_rho;
    // 4. level loop, deepest depth first.  Two score buffers: A receives this depth's MD; B holds the depth
    // below, which becomes this depth's D in place (accumulate + gamma scatter) before the pull reads it.
    PS_CUDA(ws->md_a.ensure((size_t)max_floats * sizeof(float)));
    PS_CUDA(ws->md_b.ensure((size_t)max_floats * sizeof(float)));
    float *A = ws->md_a.as<float>(), *Bm = ws->md_b.as<float>();
    const int32_t *node_list = ws->node_list.as<int32_t>();
    const PullTuning tune = g->tune;
    int32_t *d_pull_err = nullptr;
    if (tune.shape == kPullTma) {
        PS_CUDA(ws->pull_err.ensure(sizeof(int32_t)));
        d_pull_err = ws->pull_err.as<int32_t>();
        PS_CUDA(cudaMemsetAsync(d_pull_err, 0, sizeof(int32_t), st));
    }
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> marks;
    // Without profiling, the push block and the tail tile of a depth run on a second stream beside the
    // accumulate and the full-tile pull: they write other columns of A than the full tiles do.  With
    // profiling everything stays on the caller's stream, so the phase times do not overlap.
    // On a small graph the kernels are a few us long and the events between the streams cost more than they hide.
    const bool small = dg.n_active <= kSmallRows;
    const bool overlap = !ws->profiling && !small;
    auto zmask_at = [&](int32_t d) -> const uint32_t * {
        return zany[d] ? reinterpret_cast<const uint32_t *>(d_sched + o_zmask + zoff[d]) : nullptr;
    };
    if (overlap) PS_CUDA(ws->ensure_side());
    cudaStream_t ss = overlap ? ws->side : st;
    for (int32_t d = Dmax; d >= 0; --d) {
        const int32_t S = scount[d], H = hcount[d];
        // below depth 0 nobody reads the rows of nodes without out-edges (the pull and the gamma gather in-neighbours'
        // rows, the accumulate stops at n_active): they are neither pulled nor zeroed (R-MAT 2^20, one query: the widest
        // pull 3.10 -> 2.57 ms, the call 23.6 -> 20.4)
        DeviceGraph dgl = dg;
        if (d > 0) dgl.n_pieces = dg.n_pieces_active;
        const int32_t rows = d > 0 ? dg.n_active : n;
        const ColLayout La = lay[d], Lb = d + 1 <= Dmax ? lay[d + 1] : make_layout(n, 4);
        const bool side_work = H > 0 || (S > 0 && tail[d] > 0);
        if (overlap && side_work) {  // side work of this depth starts after everything before it
            PS_CUDA(cudaEventRecord(ws->ev_start, st));
            PS_CUDA(cudaStreamWaitEvent(ss, ws->ev_start, 0));
        }
        // height-2 columns: zero, then push from the grandchildren's gamma.  Zeroed: the push block, and the inherited
        // columns outside the pulled tiles (the pull writes 0 into those inside them); inherited columns are pushed
        // after the pull, below.  On a small graph the prepare launch zeroes them and all are pushed after the pull.
        const int32_t z0 = hinh[d] > 0 ? dw[d] : h0v[d];
        const bool late = small && S > 0;
        if (H > 0 && !late) {
            ph.begin(6);
            launch_zero_cols(rows, A, La, z0, rpv[d] - z0, ss);
            launch_push_h2(dg, node_list + node_off[d + 2], ncount[d + 2], t, A, La, h0v[d], 0, ss);
            ph.end();
            launches += 2;
        }
        if (S > 0) {
            ph.begin(2);  // D of this depth's dense nodes, in place in B (the MD of depth d+1)
            const int32_t np1 = p1_at[d + 1] - p1_at[d], np2 = p2_at[d + 1] - p2_at[d];
            if (np1 > 0)
                PS_CUDA(launch_accumulate(dg.n_active, Bm, Lb, rpv[d + 1], acc_src[d], d_sched + o_p1dst + p1_at[d],
                                          reinterpret_cast<const int4 *>(d_sched + o_p1src) + p1_at[d], np1,
                                          d_sched + o_p2dst + p2_at[d],
                                          reinterpret_cast<const int4 *>(d_sched + o_p2src) + p2_at[d], np2, st));
            ph.end();
            ++launches;
            ph.begin(3);  // gamma scatter into D; the spare row and the split rows zeroed for the pull
            launch_prepare_pull(dg, d + 2 <= Dmax ? node_list + node_off[d + 2] : nullptr,
                                d + 2 <= Dmax ? ncount[d + 2] : 0, t, Bm, Lb, A, La, dw[d], rows, z0,
                                late && H > 0 ? rpv[d] - z0 : 0, st);
            ph.end();
            ++launches;
            cudaEvent_t e0 = nullptr, e1 = nullptr;
            if (ws->profiling) {
                e0 = tm.get();
                e1 = tm.get();
                PS_CUDA(cudaEventRecord(e0, st));
            }
            const uint32_t *zm = zmask_at(d);
            if (tail[d] > 0) {
                if (overlap) {
                    PS_CUDA(cudaEventRecord(ws->ev_ready, st));
                    PS_CUDA(cudaStreamWaitEvent(ss, ws->ev_ready, 0));
                }
                pull_tail(dgl, tune, Bm, Lb, A, La, 32 * nfull[d], tail[d], zm ? zm + nfull[d] : nullptr, ss);
                ++launches;
            }
            PS_CUDA(pull_full(dgl, tune, Bm, Lb, A, La, nfull[d], zm, d_pull_err, &launches, st));
            if (ws->profiling) {
                PS_CUDA(cudaEventRecord(e1, st));
                marks.push_back({e0, e1});
            }
            ws->stats.probe_launches += 1;
            const int64_t edges = d > 0 ? dg.m_active : dg.m;  // of the rows pulled
            ws->stats.edge_gathers += edges * S;
            ws->stats.probe_bytes += 4.0 * edges + 16.0 * dgl.n_pieces + 4.0 * rows + 4.0 * ((double)dg.n_active + rows) * S;
        }
        if (overlap && side_work) {  // the gamma of this depth (and every later step) waits for the side work
            PS_CUDA(cudaEventRecord(ws->ev_side, ss));
            PS_CUDA(cudaStreamWaitEvent(st, ws->ev_side, 0));
        }
        if (late ? H > 0 : hinh[d] > 0) {  // push nodes in inherited columns: after the pull has written those columns as 0
            ph.begin(6);
            launch_push_h2(dg, node_list + node_off[d + 2], ncount[d + 2], t, A, La, h0v[d], late ? 2 : 1, st);
            ph.end();
            ++launches;
        }
        if (d >= 1) {
            ph.begin(7);
            launch_gamma(dg, node_list + node_off[d], ncount[d], t, qb.inv_nr, (S + H) > 0 ? A : nullptr, La, st);
            ph.end();
            ++launches;
        }
        std::swap(A, Bm);
        ws->stats.levels += 1;
    }
    float *MD0 = Bm;  // after the last swap, the super-roots' MD
    // 5. estimates: s(u, v) = MD(super-root)[v], s(u, u) = 1
    ph.begin(8);
    launch_finalize(n, B, qb.node, d_rho, scount[0] > 0 ? MD0 : nullptr, lay[0], dg.ext2int, g->cfg.shift, d_out, st);
    ph.end();
    ++launches;
    PS_CUDA(cudaGetLastError());
    int32_t pull_err = 0;
    if (d_pull_err) PS_CUDA(cudaMemcpyAsync(&pull_err, d_pull_err, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    if (pull_err) return fail(PROBESIM_E_TIMEOUT, "a TMA row gather of the pull did not complete in time");
    ph.collect(ws->stats);
    for (auto &mk : marks) {
        float ms = 0.f;
        PS_CUDA(cudaEventElapsedTime(&ms, mk.first, mk.second));
        ws->stats.probe_ms += ms;
        ws->stats.phase_ms[5] += ms;
    }
    ws->stats.kernel_launches += launches;
    return PROBESIM_OK;
}

// Walks of a planned batch (Def. 3): uploads the queries, launches the walk kernel and reads back the walk
// node count and the longest walk.
static probesim_status batch_walks(probesim_graph *g, Workspace *ws, const BatchPlan &P, QueryBatch &qb,
                                   int64_t *walk_nodes, int32_t *max_len, int64_t &launches, cudaStream_t st) {
    const int32_t L = g->cfg.l_max;
    PS_TRY(upload_batch(ws, P, qb, st));
    PS_CUDA(ws->walks.ensure(sizeof(int32_t) * std::max<int64_t>(1, (int64_t)P.W * L)));
    PS_CUDA(ws->lens.ensure(sizeof(int32_t) * std::max<int32_t>(1, P.W)));
    PS_CUDA(ws->ctr.ensure(sizeof(LaunchCounters)));
    LaunchCounters *d_ctr = ws->ctr.as<LaunchCounters>();
    PS_CUDA(cudaMemsetAsync(d_ctr, 0, sizeof(LaunchCounters), st));
    launch_walks(ws->dg, qb, P.W, L, g->t_stop, g->cfg.seed, ws->walks.as<int32_t>(), ws->lens.as<int32_t>(), false,
                 d_ctr, st);
    ++launches;
    LaunchCounters *h_ctr = ws->pin_s.as<LaunchCounters>();
    PS_CUDA(cudaMemcpyAsync(h_ctr, d_ctr, sizeof(LaunchCounters), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    *walk_nodes = (int64_t)h_ctr->walk_nodes;
    *max_len = h_ctr->max_len;
    ws->stats.walks += P.W;
    ws->stats.walk_nodes += *walk_nodes;
    return PROBESIM_OK;
}

// Randomized PROBE (Alg. 3) instances of the walks w0 .. w1-1, one per (walk, prefix length i >= 2) -- or, with
// walk_slot and t_sw, only those whose prefix's tree slot is flagged -- run level by level over frontier lists.
// Adds the member counts of the final levels into counts ([B][n], internal ids).  An allocation that
// fails sets *too_big (here: the walk range is too large) and returns PROBESIM_E_NOMEM.  A level's list holds
// list_share entries per work item; *too_short is set, with PROBESIM_E_NOMEM, when a level had more members.
static probesim_status rand_range(probesim_graph *g, Workspace *ws, const QueryBatch &qb, int32_t w0, int32_t w1,
                                  int32_t max_len, int64_t walk_nodes, const int32_t *walk_slot, const uint8_t *t_sw,
                                  int32_t *counts, double list_share, int64_t &launches, cudaStream_t st, bool *too_big,
                                  bool *too_short) {
    *too_big = *too_short = false;
    const int32_t W = w1 - w0;
    const DeviceGraph &dg = ws->dg;
    const int32_t L = g->cfg.l_max;
    if (W <= 0 || max_len < 2) return PROBESIM_OK;
    // instances: one per walk node after the first
    const int64_t ni = std::min<int64_t>(walk_nodes, (int64_t)W * (max_len - 1));
    if (ni > (int64_t)kRandCountMask) {
        *too_big = W > 1;
        return fail(PROBESIM_E_INVALID, "too many probe instances in one call");
    }
    if (ni == 0) return PROBESIM_OK;
    auto list_of = [&](int k) {
        RandList l;
        l.ent = ws->r_ent[k].as<RandEntry>();
        l.first = ws->r_first[k].as<long long>();
        l.cap = (long long)std::min(ws->r_ent[k].cap / sizeof(RandEntry), ws->r_first[k].cap / sizeof(long long));
        return l;
    };
    // the work items of the levels that a list is sized for (rand_lists.h)
    auto items_of = [&](const RandList &l) -> long long { return rand_list_items(list_share, l.cap); };
    PS_ALLOC_RANGE(ws->r_ent[0].ensure(sizeof(RandEntry) * ni));
    PS_ALLOC_RANGE(ws->r_first[0].ensure(sizeof(long long) * ni));
    // counters of levels 0 .. 255 and their checks
    PS_ALLOC_RANGE(ws->r_ctr.ensure(sizeof(unsigned long long) * 512));
    unsigned long long *d_packed = ws->r_ctr.as<unsigned long long>(), *d_check = d_packed + 256;
    PS_CUDA(cudaMemsetAsync(d_packed, 0, sizeof(unsigned long long) * 512, st));
    launch_inst_init(qb, dg, ws->lens.as<int32_t>(), w0, W, L, max_len, ws->walks.as<int32_t>(), list_of(0), d_packed,
                     d_check, walk_slot, t_sw, st);
    ++launches;
    unsigned long long *h_ctr = reinterpret_cast<unsigned long long *>(ws->pin_s.as<char>() + 32768);
    PS_CUDA(cudaMemcpyAsync(h_ctr, d_packed, sizeof(unsigned long long) * 512, cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    // Levels run several per synchronisation: a level whose members might not fit its list does nothing, so the
    // host finds the first level that waited, grows the list and goes on from there.
    int32_t group = 1;
    for (int32_t j = 0; j + 2 <= max_len;) {
        const unsigned long long packed = h_ctr[j];
        const int64_t F = (int64_t)(packed & kRandCountMask), E = (int64_t)(packed >> kRandCountBits);
        if (F == 0) break;
        const int nx = (j + 1) & 1;
        if (F > list_of(j & 1).cap) {
            *too_short = true;
            return fail(PROBESIM_E_NOMEM, "internal: a randomized PROBE level outgrew its list");
        }
        const int64_t need = std::max<int64_t>(kRandListMin, rand_list_entries(list_share, E));
        // an overflowed counter, or lists beyond the budget: a smaller walk range needs less
        if (h_ctr[256 + j] != (unsigned long long)E ||
            ((sizeof(RandEntry) + sizeof(long long)) * (size_t)need > budget_of(g, ws) / 4 && W > 1)) {
            *too_big = W > 1;
            return fail(PROBESIM_E_NOMEM, "randomized PROBE level exceeds a quarter of the memory budget");
        }
        PS_ALLOC_RANGE(ws->r_ent[nx].ensure(sizeof(RandEntry) * need));
        PS_ALLOC_RANGE(ws->r_first[nx].ensure(sizeof(long long) * need));
        const int32_t begin = j, end = std::min(max_len - 1, j + group);
        for (int32_t t = j; t < end; ++t) {
            RandLevel Lv;
            Lv.cur = list_of(t & 1);
            Lv.next = list_of((t + 1) & 1);
            Lv.max_items = items_of(Lv.next);
            Lv.packed_in = d_packed + t;
            Lv.packed_out = d_packed + t + 1;
            Lv.check_out = d_check + t + 1;
            Lv.counts = counts;
            Lv.j = t;
            launch_rand_level(dg, ws->walks.as<int32_t>(), L, qb.qid, g->cfg.seed, g->t_keep, Lv, E, st);
            ++launches;
        }
        PS_CUDA(cudaMemcpyAsync(h_ctr, d_packed, sizeof(unsigned long long) * 512, cudaMemcpyDeviceToHost, st));
        PS_CUDA(cudaStreamSynchronize(st));
        while (j < end) {  // the levels that ran: those whose work fits the list they write
            const int64_t Ej = (int64_t)(h_ctr[j] >> kRandCountBits);
            if ((h_ctr[j] & kRandCountMask) == 0 || h_ctr[256 + j] != (unsigned long long)Ej ||
                (int64_t)(h_ctr[j] & kRandCountMask) > list_of(j & 1).cap || Ej > items_of(list_of((j + 1) & 1)))
                break;
            ws->stats.edge_gathers += Ej;
            ws->stats.levels += 1;
            ++j;
        }
        if (j == begin) return fail(PROBESIM_E_CUDA, "internal: a randomized PROBE level did not run");
        group = std::min(8, 2 * group);
    }
    return PROBESIM_OK;
}

// All instances of the call (see rand_range), into ws->r_counts.  When the whole walk range does not fit, the
// walks are taken in halves, quarters, ..., each counted into a side buffer added once the range completes, so
// the integer member counts come out the same whatever the split.
static probesim_status rand_instances(probesim_graph *g, Workspace *ws, const QueryBatch &qb, int32_t B, int32_t W,
                                      int32_t max_len, int64_t walk_nodes, const int32_t *walk_slot,
                                      const uint8_t *t_sw, int64_t &launches, cudaStream_t st, bool *too_big) {
    const size_t cn = (size_t)B * g->n;
    PS_ALLOC(ws->r_counts.ensure(sizeof(int32_t) * cn));
    // Members per work item: the item (y, x) is a member's with probability sqrt(c) / |I(x)|, and the sum of 1 / |I(x)|
    // over all edges is the number of nodes with in-edges, so sqrt(c) n / m is the graph's mean.  Lists hold four times
    // that (at least one entry for eight items); a range with more members runs again with lists for every item.
    const double share = std::min(1.0, std::max(0.125, 4.0 * std::sqrt(g->cfg.c) * (double)g->n /
                                                           (double)std::max<int64_t>(1, ws->dg.m)));
    bool oom = false;
    auto range = [&](int32_t w0, int32_t w1, DevBuf &counts) -> probesim_status {
        bool too_short = false;
        PS_CUDA(cudaMemsetAsync(counts.p, 0, sizeof(int32_t) * cn, st));
        probesim_status s = rand_range(g, ws, qb, w0, w1, max_len, walk_nodes, walk_slot, t_sw, counts.as<int32_t>(),
                                       share, launches, st, &oom, &too_short);
        if (!too_short) return s;
        PS_CUDA(cudaMemsetAsync(counts.p, 0, sizeof(int32_t) * cn, st));
        return rand_range(g, ws, qb, w0, w1, max_len, walk_nodes, walk_slot, t_sw, counts.as<int32_t>(), 1.0, launches,
                          st, &oom, &too_short);
    };
    probesim_status s = range(0, W, ws->r_counts);
    if (s == PROBESIM_OK || !oom || W <= 1) {
        if (s == PROBESIM_OK) g_last_error.clear();  // a range that ran again is not an error
        if (oom) *too_big = B > 1;
        return s;
    }
    DevBuf *big[] = {&ws->r_ent[0], &ws->r_ent[1], &ws->r_first[0], &ws->r_first[1]};
    for (DevBuf *b : big) b->release();
    // the frontier engine's lists and tables (in switch mode) are done with by now: their memory goes too
    for (DevBuf *b : {&ws->f_list[0], &ws->f_list[1], &ws->f_stack, &ws->f_tasks, &ws->f_keys}) b->release();
    PS_CUDA(cudaMemsetAsync(ws->r_counts.p, 0, sizeof(int32_t) * cn, st));
    PS_ALLOC(ws->r_counts2.ensure(sizeof(int32_t) * cn));
    int32_t span = (W + 1) / 2;
    for (int32_t w0 = 0; w0 < W;) {
        const int32_t w1 = std::min(W, w0 + span);
        s = range(w0, w1, ws->r_counts2);
        if (s == PROBESIM_OK) {
            launch_add_i32(ws->r_counts.as<int32_t>(), ws->r_counts2.as<int32_t>(), (int64_t)cn, st);
            ++launches;
            w0 = w1;
        } else if (oom && span > 1) {
            span = (span + 1) / 2;
            for (DevBuf *b : big) b->release();
        } else {
            if (oom) *too_big = B > 1;
            return s;
        }
    }
    g_last_error.clear();  // the allocation failures that cut the walk range are not errors
    return PROBESIM_OK;
}

// Randomized PROBE (Alg. 3) for every probe of Alg. 1: one instance per (walk, prefix length); the estimate is
// the member count of the final levels divided by n_r.
static probesim_status run_batch_rand(probesim_graph *g, Workspace *ws, const probesim_query *q, int32_t B,
                                      float *d_out, cudaStream_t st, bool *too_big) {
    *too_big = false;
    BatchPlan P;
    PS_TRY(plan_batch(g, q, B, P));
    QueryBatch qb;
    int64_t launches = 0, walk_nodes = 0;
    int32_t max_len = 0;
    PS_TRY(batch_walks(g, ws, P, qb, &walk_nodes, &max_len, launches, st));
    PS_TRY(rand_instances(g, ws, qb, B, P.W, max_len, walk_nodes, nullptr, nullptr, launches, st, too_big));
    launch_rand_finalize(g->n, B, qb.node, ws->r_counts.as<int32_t>(), qb.inv_nr, ws->dg.ext2int, g->cfg.shift, d_out,
                         st);
    ++launches;
    PS_CUDA(cudaGetLastError());
    PS_CUDA(cudaStreamSynchronize(st));
    ws->stats.kernel_launches += launches;
    return PROBESIM_OK;
}

// Frontier engine (frontier.cu): every prefix of the batch's walk trees probed on its own with Pruning Rule 2,
// and, in PROBESIM_PROBE_SWITCH mode, the switch of Sec. 4.4 handing large probes to Alg. 3.
static probesim_status run_batch_frontier(probesim_graph *g, Workspace *ws, const probesim_query *q, int32_t B,
                                          float *d_out, cudaStream_t st, bool *too_big) {
    *too_big = false;
    const DeviceGraph &dg = ws->dg;
    const int32_t n = dg.n, L = g->cfg.l_max;
    const bool sw_mode = g->cfg.probe_mode == PROBESIM_PROBE_SWITCH;
    BatchPlan P;
    PS_TRY(plan_batch(g, q, B, P));
    int64_t max_w = 1;
    for (int32_t b = 0; b < B; ++b) {
        if (num_walks(g->cfg.c, q[b].eps, g->cfg.delta, n) > kFrontierMaxWalks)
            return fail(PROBESIM_E_INVALID, "eps too small: Pruning Rule 2 and the switch take at most 2^18 walks per query");
        max_w = std::max<int64_t>(max_w, P.base[b + 1] - P.base[b]);
    }
    if ((size_t)P.W * L * 8 > budget_of(g, ws) / 4 && B > 1) {
        *too_big = true;
        return PROBESIM_E_NOMEM;
    }
    QueryBatch qb;
    int64_t launches = 0, walk_nodes = 0;
    int32_t max_len = 0;
    PS_TRY(batch_walks(g, ws, P, qb, &walk_nodes, &max_len, launches, st));
    // reverse-reachability tree (Alg. 4) with the slot of every walk prefix
    TrieTable t;
    t.cap = next_pow2(std::max<int64_t>(1024, 2 * (walk_nodes + B) + 64));
    const size_t cap = (size_t)t.cap;
    PS_ALLOC(ws->t_key.ensure(8 * cap));
    PS_ALLOC(ws->t_node.ensure(4 * cap));
    PS_ALLOC(ws->t_parent.ensure(4 * cap));
    PS_ALLOC(ws->t_depth.ensure(4 * cap));
    PS_ALLOC(ws->t_query.ensure(4 * cap));
    PS_ALLOC(ws->t_weight.ensure(4 * cap));
    PS_ALLOC(ws->t_height.ensure(4 * cap));
    PS_ALLOC(ws->f_wslot.ensure(sizeof(int32_t) * std::max<int64_t>(1, (int64_t)P.W * L)));
    PS_ALLOC(ws->f_tsw.ensure(cap));
    t.key = ws->t_key.as<unsigned long long>();
    t.node = ws->t_node.as<int32_t>();
    t.parent = ws->t_parent.as<int32_t>();
    t.depth = ws->t_depth.as<int32_t>();
    t.query = ws->t_query.as<int32_t>();
    t.weight = ws->t_weight.as<int32_t>();
    t.height = ws->t_height.as<int32_t>();
    t.walk_slot = ws->f_wslot.as<int32_t>();
    uint8_t *t_sw = ws->f_tsw.as<uint8_t>();
    PS_CUDA(cudaMemsetAsync(t.key, 0xFF, 8 * cap, st));
    PS_CUDA(cudaMemsetAsync(t.weight, 0, 4 * cap, st));
    PS_CUDA(cudaMemsetAsync(t.height, 0, 4 * cap, st));
    PS_CUDA(cudaMemsetAsync(t_sw, 0, cap, st));
    LaunchCounters *d_ctr = ws->ctr.as<LaunchCounters>();
    // the probes: tree nodes of depth >= 2
    PS_ALLOC(ws->f_slot.ensure(sizeof(int32_t) * std::max<int64_t>(1, walk_nodes)));
    PS_ALLOC(ws->f_misc.ensure(512));
    int32_t *d_np = ws->f_misc.as<int32_t>();
    unsigned long long *d_fctr = reinterpret_cast<unsigned long long *>(ws->f_misc.as<char>() + 8);
    PS_CUDA(cudaMemsetAsync(d_np, 0, 512, st));
    t.probes = ws->f_slot.as<int32_t>();
    t.probe_count = d_np;
    launch_trie_insert(dg, qb, P.W, L, ws->walks.as<int32_t>(), ws->lens.as<int32_t>(), t, d_ctr, st);
    ++launches;
    LaunchCounters *h_ctr = ws->pin_s.as<LaunchCounters>();
    long long *h_ll = reinterpret_cast<long long *>(ws->pin_s.as<char>() + 32768);
    PS_CUDA(cudaMemcpyAsync(h_ctr, d_ctr, sizeof(LaunchCounters), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(h_ll, d_np, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    if (h_ctr->overflow) return fail(PROBESIM_E_CUDA, "internal: walk tree table overflow");
    const int32_t NP = reinterpret_cast<int32_t *>(h_ll)[0];
    ws->stats.probes += NP;
    ws->stats.tree_nodes += NP;
    // per-probe state, the estimate sums
    FrontierProbes PR;
    PR.P = NP;
    const size_t np1 = (size_t)std::max(1, NP);
    PS_ALLOC(ws->f_pr32.ensure(sizeof(int32_t) * 6 * np1));
    PS_ALLOC(ws->f_pr64.ensure(sizeof(long long) * 6 * np1));
    PR.slot = ws->f_slot.as<int32_t>();
    int32_t *i32 = ws->f_pr32.as<int32_t>();
    PR.anc = i32, PR.lev = i32 + np1, PR.ex = i32 + 2 * np1, PR.state = i32 + 3 * np1, PR.cls = i32 + 4 * np1;
    PR.nt = reinterpret_cast<uint32_t *>(i32 + 5 * np1);
    long long *i64 = ws->f_pr64.as<long long>();
    PR.rsize = i64 + 4 * np1, PR.roff = i64 + 5 * np1;
    auto of_parity = [&](int cur) {  // this level's segments and counters and the next level's change places
        FrontierProbes p = PR;
        p.packed = reinterpret_cast<unsigned long long *>(i64 + cur * np1);
        p.packed_nx = reinterpret_cast<unsigned long long *>(i64 + (cur ^ 1) * np1);
        p.beg = i64 + (2 + cur) * np1;
        p.beg_nx = i64 + (2 + (cur ^ 1)) * np1;
        return p;
    };
    const size_t accn = (size_t)B * n;
    PS_ALLOC(ws->f_acc.ensure(sizeof(unsigned long long) * accn));
    PS_CUDA(cudaMemsetAsync(ws->f_acc.p, 0, sizeof(unsigned long long) * accn, st));
    // host tables: thr[w] = floor(c0 * w * n) in FP64 (the switch compares the integer out-degree sum with it),
    // pw[k] = sqrt(c)^k rounded to FP32 (Rule 2's factor)
    const size_t nthr = sw_mode ? (size_t)max_w + 1 : 0;
    const size_t tab_bytes = 256 * sizeof(float) + nthr * sizeof(long long);
    PS_ALLOC(ws->f_tab.ensure(tab_bytes));
    PS_ALLOC(ws->pin_q.ensure(tab_bytes));
    {
        char *h = ws->pin_q.as<char>();
        float *pw = reinterpret_cast<float *>(h);
        const double sc = std::sqrt(g->cfg.c);
        for (int k = 0; k < 256; ++k) pw[k] = (float)std::pow(sc, (double)k);
        long long *thr = reinterpret_cast<long long *>(h + 256 * sizeof(float));
        for (size_t w = 0; w < nthr; ++w) {
            const double x = std::floor((double)g->cfg.c0 * (double)w * (double)n);
            thr[w] = x >= 9.0e18 ? (long long)9000000000000000000ll : (long long)x;
        }
        PS_CUDA(cudaMemcpyAsync(ws->f_tab.p, h, tab_bytes, cudaMemcpyHostToDevice, st));
    }
    const float *d_pw = ws->f_tab.as<float>();
    const long long *d_thr = sw_mode ? reinterpret_cast<const long long *>(ws->f_tab.as<char>() + 256 * sizeof(float)) : nullptr;
    // The deterministic rounds work on probe ranges [p0, p1) at a level j.  A range whose next frontiers, global tables or
    // task lists might not fit their part of the budget keeps as many of its first probes as the bounds allow and defers the
    // others, with their level-j segments, to a stack; they resume once the kept probes have run out.  Every probe's
    // last-level pushes land in the estimate exactly once, whatever the split.
    const long long slot_cap =
        std::max<long long>((long long)n, (long long)(budget_of(g, ws) / 4 / sizeof(FrontierSlot)));
    const long long list_cap =
        std::max<long long>((long long)n, (long long)(budget_of(g, ws) / 8 / sizeof(FrontierEntry)));
    // tasks of a level (a last-level or single-entry probe has one per kFrChunk items and no next frontier or table to be
    // held back by); one probe's fit n or 2^31 / kFrChunk, and a class's number is a grid size
    const long long task_cap = std::min<long long>(
        ((long long)1 << 31) - 1,
        std::max<long long>((long long)n, (long long)(budget_of(g, ws) / 16 / sizeof(FrontierTask))));
    struct Range {
        int32_t p0, p1, j;
        int cur;
        bool on_stack;  // segments in the stack buffer, else in list cur
        long long at;   // on_stack: the stack's height below them
    };
    std::vector<Range> stack;
    Range R{0, NP, 0, 0, false, 0};
    long long stack_top = 0;
    unsigned long long *d_tot = d_fctr + 1, *d_cursor = d_tot + kFrTotals, *d_top = d_cursor + kFrTotals;
    unsigned long long *h_tot = reinterpret_cast<unsigned long long *>(h_ll);
    PS_ALLOC(ws->f_list[0].ensure(sizeof(FrontierEntry) * np1));
    launch_fr_init(t, of_parity(0), dg.out_off, d_pw, g->cfg.eps_p, ws->f_list[0].as<FrontierEntry>(), st);
    ++launches;
    bool live = NP > 0;
    for (;;) {
        if (!live) {  // the range ran out: resume the last deferred one
            if (stack.empty()) break;
            R = stack.back();
            stack.pop_back();
            ws->stats.deferred += 1;
            live = true;
        }
        const FrontierEntry *src = R.on_stack ? ws->f_stack.as<FrontierEntry>() : ws->f_list[R.cur].as<FrontierEntry>();
        PS_CUDA(cudaMemsetAsync(d_tot, 0, sizeof(unsigned long long) * 2 * kFrTotals, st));  // and the cursors
        if (d_thr && g->cfg.eps_p <= 0.f) {
            launch_fr_check(dg, t, of_parity(R.cur), R.p0, R.p1, R.j, src, d_thr, t_sw, st);
            ++launches;
        }
        launch_fr_plan(t, of_parity(R.cur), R.p0, R.p1, R.j, n, d_thr, t_sw, d_tot, st);
        ++launches;
        PS_CUDA(cudaMemcpyAsync(h_tot, d_tot, sizeof(unsigned long long) * kFrTotals, cudaMemcpyDeviceToHost, st));
        PS_CUDA(cudaStreamSynchronize(st));
        const long long D = (long long)h_tot[kFrTotD], G = (long long)h_tot[kFrTotGlobal];
        if (h_tot[kFrTotItems] == 0) {  // nothing left to push: every probe of the range ended, switched or was pruned
            if (R.on_stack) stack_top = R.at;
            live = false;
            continue;
        }
        long long nt = 0;
        for (int c = kFrNone + 1; c < kFrClasses; ++c) nt += (long long)h_tot[c];
        if ((D > list_cap || G > slot_cap || nt > task_cap) && R.p1 - R.p0 > 1) {  // defer the range's last probes
            const double keep = 0.9 * std::min({D > 0 ? (double)list_cap / (double)D : 1.0,
                                                G > 0 ? (double)slot_cap / (double)G : 1.0,
                                                nt > 0 ? (double)task_cap / (double)nt : 1.0});
            const int32_t pm = R.p0 + std::max(1, (int32_t)std::min<double>(keep * (R.p1 - R.p0), R.p1 - R.p0 - 1));
            Range tail{pm, R.p1, R.j, R.cur, true, R.on_stack ? R.at : stack_top};
            if (!R.on_stack) {
                const long long cnt = (long long)h_tot[kFrTotEntries];  // of the whole range: enough
                PS_ALLOC(ws->f_stack.grow(sizeof(FrontierEntry) * (stack_top + cnt), sizeof(FrontierEntry) * stack_top,
                                          st));
                h_tot[0] = (unsigned long long)stack_top;
                PS_CUDA(cudaMemcpyAsync(d_top, h_tot, sizeof(unsigned long long), cudaMemcpyHostToDevice, st));
                launch_fr_defer(of_parity(R.cur), pm, R.p1, src, ws->f_stack.as<FrontierEntry>(), d_top, st);
                ++launches;
                PS_CUDA(cudaMemcpyAsync(h_tot, d_top, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
                PS_CUDA(cudaStreamSynchronize(st));
                stack_top = (long long)h_tot[0];
            }
            // a range read from the stack leaves its tail where it is: the tail then owns the space down to R.at
            stack.push_back(tail);
            if (R.on_stack) R.at = stack_top;
            R.p1 = pm;
            continue;
        }
        ws->stats.edge_gathers += (int64_t)h_tot[kFrTotItems];
        ws->stats.levels += 1;
        if (D > 0) ws->stats.table_passes += 1;
        ws->stats.max_table_slots = std::max<int64_t>(ws->stats.max_table_slots, (int64_t)h_tot[kFrTotSlots]);
        FrontierBases base;
        for (int c = kFrLast; c < kFrSweep; ++c) base.at[c + 1] = base.at[c] + (long long)h_tot[c];
        const int nx = R.cur ^ 1;
        PS_ALLOC(ws->f_list[nx].ensure(sizeof(FrontierEntry) * std::max<long long>(1, D)));
        PS_ALLOC(ws->f_tasks.ensure(sizeof(FrontierTask) * std::max<long long>(1, nt)));
        if (G > 0) {
            bool fresh = false;
            PS_ALLOC(ws->f_keys.ensure(sizeof(FrontierSlot) * G, &fresh));
            const bool clear = fresh || !ws->f_table_clean;  // new memory, or a failed call left slots behind
            ws->f_table_clean = false;                       // until this level's sweep has emptied its slots
            if (clear) PS_CUDA(cudaMemsetAsync(ws->f_keys.p, 0, ws->f_keys.cap, st));
        }
        launch_fr_tasks(of_parity(R.cur), R.p0, R.p1, n, base, d_cursor, ws->f_tasks.as<FrontierTask>(), st);
        ++launches;
        FrontierLevel a;
        a.tasks = ws->f_tasks.as<FrontierTask>();
        a.src = src;
        a.dst = ws->f_list[nx].as<FrontierEntry>();
        a.tab = ws->f_keys.as<FrontierSlot>();
        a.acc = ws->f_acc.as<unsigned long long>();
        a.pw = d_pw;
        a.eps_p = g->cfg.eps_p;
        a.j = R.j;
        a.one_query = B == 1;
        PS_CUDA(launch_fr_level(dg, t, of_parity(R.cur), a, base, h_tot, st, &launches));
        PS_CUDA(cudaGetLastError());
        if (G > 0) ws->f_table_clean = true;
        if (R.on_stack) stack_top = R.at;
        R = Range{R.p0, R.p1, R.j + 1, nx, false, 0};
    }
    launch_fr_count_switched(PR, d_fctr, st);
    PS_CUDA(cudaMemcpyAsync(h_ll, d_fctr, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    const int64_t switched = h_ll[0];
    ws->stats.switched += switched;
    // Sec. 4.4: Alg. 3 for every walk through a switched tree node
    const int32_t *counts = nullptr;
    if (switched > 0) {
        PS_TRY(rand_instances(g, ws, qb, B, P.W, max_len, walk_nodes, t.walk_slot, t_sw, launches, st, too_big));
        counts = ws->r_counts.as<int32_t>();
    }
    launch_fr_finalize(n, B, qb.node, ws->f_acc.as<unsigned long long>(), counts, qb.inv_nr, dg.ext2int, g->cfg.shift,
                       d_out, st);
    ++launches;
    PS_CUDA(cudaGetLastError());
    PS_CUDA(cudaStreamSynchronize(st));
    ws->stats.kernel_launches += launches;
    return PROBESIM_OK;
}

// Runs all nq queries, splitting batches that do not fit the workspace budget.
static probesim_status run_queries(probesim_graph *g, Workspace *ws, const probesim_query *q, int32_t nq, float *d_out,
                                   cudaStream_t st) {
    int32_t done = 0;
    int32_t chunk = nq;
    while (done < nq) {
        const int32_t B = std::min(chunk, nq - done);
        bool too_big = false;
        float *out = d_out + (int64_t)done * g->n;
        probesim_status s;
        if (g->cfg.probe_mode == PROBESIM_PROBE_RANDOMIZED)
            s = run_batch_rand(g, ws, q + done, B, out, st, &too_big);
        else if (g->cfg.probe_mode == PROBESIM_PROBE_SWITCH || g->cfg.eps_p > 0.f)
            s = run_batch_frontier(g, ws, q + done, B, out, st, &too_big);
        else
            s = run_batch(g, ws, q + done, B, out, st, &too_big);
        if (s == PROBESIM_OK) {
            done += B;
            continue;
        }
        if (too_big && B > 1) {
            chunk = std::max(1, B / 2);
            continue;
        }
        return s;
    }
    if (chunk < nq) g_last_error.clear();  // the budget messages of batches that were split are not errors
    return PROBESIM_OK;
}

probesim_status ps::check_queries(const probesim_graph *g, const probesim_query *q, int32_t nq, bool topk,
                                     int32_t kmax) {
    if (!q || nq <= 0) return fail(PROBESIM_E_INVALID, "queries: null pointer or nq <= 0");
    if (nq > 65535) return fail(PROBESIM_E_INVALID, "at most 65535 queries per call");
    for (int32_t i = 0; i < nq; ++i) {
        if (q[i].node < 0 || q[i].node >= g->n) return fail(PROBESIM_E_RANGE, "query node outside [0, n)");
        if (!(q[i].eps > 0.0 && q[i].eps < 1.0)) return fail(PROBESIM_E_INVALID, "query eps must lie in (0, 1)");
        if (topk && (q[i].k < 1 || q[i].k > kmax)) return fail(PROBESIM_E_INVALID, "query k must lie in [1, kmax]");
    }
    return PROBESIM_OK;
}

// ------------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------------
extern "C" {

const char *probesim_last_error(void) { return g_last_error.c_str(); }

probesim_status probesim_config_default(probesim_config *cfg) {
    if (!cfg) return fail(PROBESIM_E_INVALID, "cfg is null");
    cfg->c = 0.6;
    cfg->delta = 0.01;
    cfg->l_max = 64;
    cfg->eps_p = 0.f;
    cfg->c0 = 1.f;
    cfg->probe_mode = PROBESIM_PROBE_DETERMINISTIC;
    cfg->seed = 3;
    cfg->shift = 0.f;
    return PROBESIM_OK;
}

probesim_status probesim_split_error(double eps_a, double c, int32_t shift, probesim_error_split *out) {
    if (!out) return fail(PROBESIM_E_INVALID, "out is null");
    if (!(eps_a > 0.0 && eps_a < 1.0)) return fail(PROBESIM_E_INVALID, "eps_a must lie in (0, 1)");
    if (!(c > 0.0 && c < 1.0)) return fail(PROBESIM_E_INVALID, "c must lie in (0, 1)");
    const double sc = std::sqrt(c);
    const double eps = eps_a / 2.0, rest = eps_a / 2.0;
    // Rule 1: error in [0, sqrt(c)^l_max] per walk, centred by the shift
    const double eps_t = shift ? rest : rest / 2.0;
    int32_t l_max = (int32_t)std::ceil(std::log(eps_t) / std::log(sc));
    l_max = std::max(1, std::min(255, l_max));
    // Rule 2: (1 + eps) * E[l (l - 1) / 2] * eps_p = rest / 2
    const double per_walk = sc / ((1.0 - sc) * (1.0 - sc));
    double ep = rest / 2.0 / ((1.0 + eps) * per_walk);
    float epf = (float)ep;
    if ((double)epf > ep) epf = std::nextafter(epf, 0.f);
    out->eps = eps;
    out->eps_t = eps_t;
    out->l_max = l_max;
    out->eps_p = epf;
    out->shift = shift ? (float)(eps_t / 2.0) : 0.f;
    const double r1 = std::pow(sc, (double)l_max) * (shift ? 0.5 : 1.0);
    out->bound = eps + (1.0 + eps) * per_walk * (double)epf + r1;
    out->bound_paper = eps + (1.0 + eps) / (1.0 - sc) * (double)epf + r1;
    return PROBESIM_OK;
}

probesim_status probesim_graph_create(int32_t n, const int32_t *src, const int32_t *dst, int64_t m,
                                      const probesim_config *cfg, void *stream, probesim_graph **out) {
    g_last_error.clear();
    if (!out) return fail(PROBESIM_E_INVALID, "out is null");
    *out = nullptr;
    if (n < 1) return fail(PROBESIM_E_INVALID, "n must be >= 1");
    if (m < 0 || m >= ((int64_t)1 << 31)) return fail(PROBESIM_E_INVALID, "m must lie in [0, 2^31)");
    if (m > 0 && (!src || !dst)) return fail(PROBESIM_E_INVALID, "src/dst is null");
    probesim_config c;
    if (cfg) c = *cfg; else probesim_config_default(&c);
    if (!(c.c > 0.0 && c.c < 1.0)) return fail(PROBESIM_E_INVALID, "c must lie in (0, 1)");
    if (!(c.delta > 0.0 && c.delta < 1.0)) return fail(PROBESIM_E_INVALID, "delta must lie in (0, 1)");
    if (c.l_max < 1 || c.l_max > 255) return fail(PROBESIM_E_INVALID, "l_max must lie in [1, 255]");
    if (!(c.eps_p >= 0.f) || !(c.c0 >= 0.f) || !(c.shift >= 0.f))
        return fail(PROBESIM_E_INVALID, "eps_p, c0 and shift must be >= 0");
    if (c.probe_mode < 0 || c.probe_mode > 2) return fail(PROBESIM_E_INVALID, "unknown probe_mode");
    probesim_graph *g = new (std::nothrow) probesim_graph();
    if (!g) return fail(PROBESIM_E_NOMEM, "host allocation failed");
    g->cfg = c;
    g->t_stop = threshold_stop(c.c);
    g->t_keep = threshold_keep(c.c);
    cudaGetDevice(&g->device);
    size_t fr = 0, tot = 0;
    cudaMemGetInfo(&fr, &tot);
    g->budget0 = (size_t)(0.6 * (double)tot);
    g->budget = g->budget0;
    if (g->ws0.pin_s.ensure(65536) != cudaSuccess) {
        delete g;
        return fail(PROBESIM_E_NOMEM, "pinned host allocation failed");
    }
    probesim_status s;
    {   // the edge list on the device (copied there when the caller's arrays are on the host), then the build
        const bool on_dev = m == 0 || (is_device_ptr(src) && is_device_ptr(dst));
        DevBuf staged;
        const int32_t *d_src = src, *d_dst = dst;
        s = PROBESIM_OK;
        if (!on_dev) {
            cudaError_t e = staged.ensure(2 * sizeof(int32_t) * (size_t)m);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(staged.p, src, sizeof(int32_t) * m, cudaMemcpyDefault, (cudaStream_t)stream);
            if (e == cudaSuccess)
                e = cudaMemcpyAsync(staged.as<int32_t>() + m, dst, sizeof(int32_t) * m, cudaMemcpyDefault,
                                    (cudaStream_t)stream);
            if (e != cudaSuccess)
                s = fail(e == cudaErrorMemoryAllocation ? PROBESIM_E_NOMEM : PROBESIM_E_CUDA,
                         std::string("staging the edge list: ") + cudaGetErrorString(e));
            d_src = staged.as<int32_t>();
            d_dst = staged.as<int32_t>() + m;
        }
        if (s == PROBESIM_OK) s = build_graph(g, n, d_src, d_dst, m, (cudaStream_t)stream);
        cudaStreamSynchronize((cudaStream_t)stream);
        staged.release();
    }
    if (s != PROBESIM_OK) {
        probesim_graph_destroy(g);
        return s;
    }
    {   // update batches allocate store versions from the device's stream-ordered pool: let it keep about three
        // versions' worth of memory between updates instead of returning it to the driver at every synchronisation
        cudaMemPool_t pool;
        if (cudaDeviceGetDefaultMemPool(&pool, g->device) == cudaSuccess) {
            const std::shared_ptr<StoreVersion> v = g->current();
            uint64_t keep = 0;
            for (DevBuf *b : {&v->in_off, &v->in_col, &v->out_off, &v->out_col, &v->w, &v->rec, &v->piece_v, &v->piece_beg,
                              &v->piece_len, &v->split_v})
                keep += b->cap;
            keep *= 3;
            uint64_t cur = 0;
            cudaMemPoolGetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &cur);
            if (cur < keep) cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
        }
        cudaGetLastError();
    }
    *out = g;
    return PROBESIM_OK;
}

probesim_status probesim_pair_mc(probesim_graph *g, const int32_t *u, const int32_t *v, const uint32_t *key_u,
                                 const uint32_t *key_v, int32_t npairs, int64_t r, int64_t *meets, float *est,
                                 void *stream) {
    if (!g || !u || !v || !key_u || !key_v || !meets) return fail(PROBESIM_E_INVALID, "null argument");
    if (npairs < 1 || npairs > 65535) return fail(PROBESIM_E_INVALID, "npairs must lie in [1, 65535]");
    if (r < 1 || r >= ((int64_t)1 << 32)) return fail(PROBESIM_E_INVALID, "r must lie in [1, 2^32)");
    for (int32_t i = 0; i < npairs; ++i)
        if (u[i] < 0 || u[i] >= g->n || v[i] < 0 || v[i] >= g->n) return fail(PROBESIM_E_RANGE, "node outside [0, n)");
    std::lock_guard<std::mutex> lk(g->mu);
    const std::shared_ptr<StoreVersion> snap = g->current();
    g_last_error.clear();
    Workspace *ws = &g->ws0;
    cudaStream_t st = (cudaStream_t)stream;
    const size_t words = 4 * (size_t)npairs;
    PS_CUDA(ws->pm_in.ensure(sizeof(int32_t) * words));
    PS_CUDA(ws->pm_meets.ensure(sizeof(unsigned long long) * npairs));
    PS_CUDA(ws->pin_q.ensure(std::max(sizeof(int32_t) * words, sizeof(unsigned long long) * npairs)));
    int32_t *h = ws->pin_q.as<int32_t>();
    std::memcpy(h, u, sizeof(int32_t) * npairs);
    std::memcpy(h + npairs, v, sizeof(int32_t) * npairs);
    std::memcpy(h + 2 * npairs, key_u, sizeof(uint32_t) * npairs);
    std::memcpy(h + 3 * npairs, key_v, sizeof(uint32_t) * npairs);
    int32_t *d = ws->pm_in.as<int32_t>();
    PS_CUDA(cudaMemcpyAsync(d, h, sizeof(int32_t) * words, cudaMemcpyHostToDevice, st));
    unsigned long long *dm = ws->pm_meets.as<unsigned long long>();
    PS_CUDA(cudaMemsetAsync(dm, 0, sizeof(unsigned long long) * npairs, st));
    launch_pair_mc(snap->dg, d, d + npairs, reinterpret_cast<const uint32_t *>(d + 2 * npairs),
                   reinterpret_cast<const uint32_t *>(d + 3 * npairs), npairs, r, g->cfg.l_max, g->cfg.seed, g->t_stop,
                   dm, st);
    PS_CUDA(cudaGetLastError());
    std::vector<unsigned long long> hm(npairs);
    PS_CUDA(cudaMemcpyAsync(hm.data(), dm, sizeof(unsigned long long) * npairs, cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    std::vector<int64_t> m64(hm.begin(), hm.end());
    std::vector<float> e(npairs);
    for (int32_t i = 0; i < npairs; ++i) e[i] = u[i] == v[i] ? 1.f : (float)((double)hm[i] / (double)r);
    if (is_device_ptr(meets)) PS_CUDA(cudaMemcpy(meets, m64.data(), sizeof(int64_t) * npairs, cudaMemcpyHostToDevice));
    else std::memcpy(meets, m64.data(), sizeof(int64_t) * npairs);
    if (est) {
        if (is_device_ptr(est)) PS_CUDA(cudaMemcpy(est, e.data(), sizeof(float) * npairs, cudaMemcpyHostToDevice));
        else std::memcpy(est, e.data(), sizeof(float) * npairs);
    }
    return PROBESIM_OK;
}

probesim_status probesim_set_memory_budget(probesim_graph *g, double bytes) {
    if (!g) return fail(PROBESIM_E_INVALID, "graph is null");
    if (!(bytes >= 0.0)) return fail(PROBESIM_E_INVALID, "bytes must be >= 0");
    std::lock_guard<std::mutex> lk(g->mu);
    g->budget = bytes > 0.0 ? (size_t)bytes : g->budget0;
    return PROBESIM_OK;
}

probesim_status probesim_graph_destroy(probesim_graph *g) {
    if (!g) return PROBESIM_OK;
    g->store.reset();
    DevBuf *bufs[] = {&g->ext2int, &g->int2ext, &g->u_batch, &g->u_valid,
                      &g->u_vpre, &g->u_delta, &g->u_deg, &g->u_part, &g->u_hist, &g->u_bounds,
                      &g->u_raw, &g->u_keys[0], &g->u_keys[1], &g->u_keys[2], &g->u_sort};
    for (DevBuf *b : bufs) b->release();
    if (g->u_ready) cudaEventDestroy(g->u_ready);
    if (g->u_stream) cudaStreamDestroy(g->u_stream);
    g->ws0.release();
    delete g;
    return PROBESIM_OK;
}

probesim_status probesim_graph_info(const probesim_graph *g, int32_t *n, int64_t *m, uint64_t *epoch) {
    if (!g) return fail(PROBESIM_E_INVALID, "graph is null");
    const std::shared_ptr<StoreVersion> v = const_cast<probesim_graph *>(g)->current();
    if (n) *n = g->n;
    if (m) *m = v->dg.m;
    if (epoch) *epoch = v->epoch;
    return PROBESIM_OK;
}

}  // extern "C"

// The batch runs on the graph's own stream of the highest priority, so it does not queue behind a query that the caller's
// stream already holds: on one stream it ended when the query did (65,536 nodes, a query of 320 ms: an update of 5,000
// edges took 190 ms beside it, now 1.9).  Only edges in device or pinned memory make it wait for the caller's stream,
// which may still be writing them.  The call returns when the batch is done, so nothing of the caller's is used after
// that.
probesim_status ps::apply_updates(probesim_graph *g, const int32_t *src, const int32_t *dst, int64_t k, bool insert,
                                  int64_t *applied, cudaStream_t caller) {
    if (!g) return fail(PROBESIM_E_INVALID, "graph is null");
    if (k < 0 || (k > 0 && (!src || !dst))) return fail(PROBESIM_E_INVALID, "bad update batch");
    std::lock_guard<std::mutex> lk(g->update_mu);
    g_last_error.clear();
    const int32_t n = g->n;
    const std::shared_ptr<StoreVersion> old = g->current();  // read only; queries may be reading it too
    auto unchanged = [&]() -> probesim_status {  // nothing but the epoch: the next version shares the arrays
        auto nv = std::make_shared<StoreVersion>();
        nv->base = old;
        nv->dg = old->dg;
        nv->epoch = old->epoch + 1;
        g->publish(nv);
        if (applied) *applied = 0;
        return PROBESIM_OK;
    };
    if (k == 0) return unchanged();
    cudaStreamCaptureStatus capturing = cudaStreamCaptureStatusNone;
    PS_CUDA(cudaStreamIsCapturing(caller, &capturing));
    if (capturing != cudaStreamCaptureStatusNone)
        return fail(PROBESIM_E_CUDA, "an update batch synchronises and cannot be captured");
    PS_CUDA(g->ensure_update_stream());
    const cudaStream_t st = g->u_stream;
    if (!is_plain_host_ptr(src) || !is_plain_host_ptr(dst)) {
        PS_CUDA(cudaEventRecord(g->u_ready, caller));
        PS_CUDA(cudaStreamWaitEvent(st, g->u_ready, 0));
    }
    // the batch on the device, without loops and repeats, in the two row orders (sorted there: the host's two sorts of
    // 10,000 edges took 0.7 ms of an update)
    const int32_t *d_src = src, *d_dst = dst;
    if (!is_device_ptr(src) || !is_device_ptr(dst)) {
        PS_CUDA(g->u_raw.ensure(2 * sizeof(int32_t) * (size_t)k));
        PS_CUDA(cudaMemcpyAsync(g->u_raw.p, src, sizeof(int32_t) * (size_t)k, cudaMemcpyDefault, st));
        PS_CUDA(cudaMemcpyAsync(g->u_raw.as<int32_t>() + k, dst, sizeof(int32_t) * (size_t)k, cudaMemcpyDefault, st));
        d_src = g->u_raw.as<int32_t>();
        d_dst = d_src + k;
    }
    int bs = 1;  // bits of a node id
    while (((int64_t)(n - 1) >> bs) > 0) ++bs;
    const int64_t ntiles = radix_tiles(k);
    PS_CUDA(g->u_hist.ensure(sizeof(unsigned long long) * (4 * (kPiece + 1) + 2)));
    for (DevBuf &b : g->u_keys) PS_CUDA(b.ensure(8 * (size_t)(k + 1)));
    PS_CUDA(g->u_sort.ensure(8 * (size_t)(2 * 256 * ntiles + 1)));
    PS_CUDA(g->u_part.ensure(sizeof(long long) * scan64_partials_needed(std::max<int64_t>({k, n, 256 * ntiles}))));
    uint64_t *ka = g->u_keys[0].as<uint64_t>(), *kb = g->u_keys[1].as<uint64_t>(), *kc = g->u_keys[2].as<uint64_t>();
    long long *cnt = g->u_sort.as<long long>(), *coff = cnt + 256 * ntiles, *part = g->u_part.as<long long>();
    int32_t *d_bad = g->u_hist.as<int32_t>();
    const int32_t *ext2int = g->ext2int.as<int32_t>();
    const uint64_t end_key = (uint64_t)1 << 2 * bs;
    PS_CUDA(cudaMemsetAsync(d_bad, 0, sizeof(int32_t), st));
    launch_batch_keys(d_src, d_dst, k, n, bs, ext2int, ka, d_bad, st);
    uint64_t *sorted = radix_sort_u64(ka, kb, k, 0, 2 * bs + 1, cnt, coff, part, st);
    long long *pre = reinterpret_cast<long long *>(sorted == ka ? kb : ka);
    launch_build_flags(sorted, k, end_key, pre, st);
    launch_scan64(pre, k, part, pre, st);  // in place: pre[k] = the number of distinct edges
    launch_build_compact(sorted, k, end_key, pre, kc, st);
    long long hk = 0;
    int32_t bad = 0;
    PS_CUDA(cudaMemcpyAsync(&bad, d_bad, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(&hk, pre + k, sizeof(long long), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaGetLastError());
    PS_CUDA(cudaStreamSynchronize(st));
    if (bad) return fail(PROBESIM_E_RANGE, "edge id outside [0, n)");
    const int64_t K = (int64_t)hk;
    if (K == 0) return unchanged();
    PS_CUDA(g->u_batch.ensure(sizeof(int32_t) * 5 * K));
    int32_t *db = g->u_batch.as<int32_t>();
    launch_batch_in(kc, K, bs, ext2int, db, db + K, db + 2 * K, ka, st);
    const uint64_t *osorted = radix_sort_u64(ka, kb, K, bs, 2 * bs, cnt, coff, part, st);  // they start in destination order
    launch_batch_out(osorted, K, bs, db + 3 * K, db + 4 * K, st);
    const DeviceGraph &dg = old->dg;
    auto nv = std::make_shared<StoreVersion>();  // the next version, built beside the current one
    PS_CUDA(g->u_bounds.ensure(upd_bounds_bytes(K)));
    PS_CUDA(g->u_valid.ensure(sizeof(long long) * 2 * K));
    PS_CUDA(g->u_vpre.ensure(sizeof(long long) * 2 * (K + 1)));
    PS_CUDA(g->u_delta.ensure(sizeof(long long) * 2 * (size_t)n));
    PS_CUDA(g->u_deg.ensure(sizeof(long long) * 2 * ((size_t)n + 1)));
    UpdateBatchArgs a;
    a.k = K;
    a.in_dst = db; a.in_src = db + K; a.in_src_ext = db + 2 * K; a.out_src = db + 3 * K; a.out_dst = db + 4 * K;
    a.in_valid = g->u_valid.as<long long>();
    a.out_valid = a.in_valid + K;
    long long *in_vpre = g->u_vpre.as<long long>(), *out_vpre = in_vpre + (K + 1);
    a.in_vpre = in_vpre;
    a.out_vpre = out_vpre;
    a.insert = insert;
    long long *in_delta = g->u_delta.as<long long>(), *out_delta = in_delta + n;
    PS_CUDA(cudaMemsetAsync(in_delta, 0, sizeof(long long) * 2 * (size_t)n, st));
    launch_upd_mark(dg, a, in_delta, out_delta, st);
    launch_scan64(a.in_valid, K, g->u_part.as<long long>(), in_vpre, st);
    launch_scan64(a.out_valid, K, g->u_part.as<long long>(), out_vpre, st);
    // new offsets
    long long *deg = g->u_deg.as<long long>(), *deg_out = deg + (n + 1);
    DevBuf &n_in_off = nv->in_off, &n_out_off = nv->out_off, &n_in_col = nv->in_col, &n_out_col = nv->out_col;
    PS_CUDA(n_in_off.alloc_pooled(sizeof(int64_t) * ((size_t)n + 1), st));
    PS_CUDA(n_out_off.alloc_pooled(sizeof(int64_t) * ((size_t)n + 1), st));
    launch_upd_degrees(n, dg.in_off, in_delta, deg, st);
    launch_scan64(deg, n, g->u_part.as<long long>(), n_in_off.as<long long>(), st);
    launch_upd_degrees(n, dg.out_off, out_delta, deg_out, st);
    launch_scan64(deg_out, n, g->u_part.as<long long>(), n_out_off.as<long long>(), st);
    long long hm[3] = {0, 0, 0};
    PS_CUDA(cudaMemcpyAsync(&hm[0], n_in_off.as<long long>() + n, sizeof(long long), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(&hm[1], n_out_off.as<long long>() + n, sizeof(long long), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(&hm[2], in_vpre + K, sizeof(long long), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    const int64_t m2 = hm[0];
    if (m2 != hm[1]) return fail(PROBESIM_E_CUDA, "internal: in- and out-lists disagree after the update");
    if (m2 >= ((int64_t)1 << 31)) return fail(PROBESIM_E_INVALID, "edge count would reach 2^31");
    PS_CUDA(n_in_col.alloc_pooled(sizeof(int32_t) * std::max<int64_t>(1, m2), st));
    PS_CUDA(n_out_col.alloc_pooled(sizeof(int32_t) * std::max<int64_t>(1, m2), st));
    launch_upd_rows(dg, a, true, n_in_off.as<long long>(), n_in_col.as<int32_t>(), g->u_bounds.p, st);
    launch_upd_rows(dg, a, false, n_out_off.as<long long>(), n_out_col.as<int32_t>(), g->u_bounds.p, st);
    // w and pieces of the new in-lists
    const int64_t cap_pieces = (int64_t)n + m2 / kPiece + 1;
    DevBuf &n_pv = nv->piece_v, &n_pb = nv->piece_beg, &n_pl = nv->piece_len, &n_split = nv->split_v;
    PS_CUDA(n_pv.alloc_pooled(sizeof(int32_t) * cap_pieces, st));
    PS_CUDA(n_pb.alloc_pooled(sizeof(int64_t) * cap_pieces, st));
    PS_CUDA(n_pl.alloc_pooled(sizeof(int32_t) * cap_pieces, st));
    PS_CUDA(n_split.alloc_pooled(sizeof(int32_t) * (size_t)n, st));
    PS_CUDA(nv->w.alloc_pooled(sizeof(float) * (size_t)n, st));
    PS_CUDA(nv->rec.alloc_pooled(sizeof(int4) * (size_t)n, st));
    launch_upd_w(n, n_in_off.as<long long>(), n_in_col.as<int32_t>(), (float)std::sqrt(g->cfg.c),
                 g->int2ext.as<int32_t>(), dg.rec_shift, nv->w.as<float>(), nv->rec.as<int4>(), deg, st);
    const int nb = 2 * (kPiece + 1);
    unsigned long long *hist = g->u_hist.as<unsigned long long>(), *cursor = hist + nb, *nsplit = cursor + nb;
    // the rows with out-edges after the batch (the last slot of the histogram buffer is free)
    int32_t *d_active = reinterpret_cast<int32_t *>(nsplit + 1);
    PS_CUDA(cudaMemsetAsync(d_active, 0, sizeof(int32_t), st));
    launch_active_rows(n_out_off.as<int64_t>(), n, d_active, st);
    launch_upd_pieces(n, n_in_off.as<long long>(), d_active, hist, cursor, n_split.as<int32_t>(), nsplit,
                      n_pv.as<int32_t>(), n_pb.as<int64_t>(), n_pl.as<int32_t>(), st);
    std::vector<unsigned long long> hh(nb + 1);
    int32_t n_active = 0;
    PS_CUDA(cudaMemcpyAsync(hh.data(), hist, sizeof(unsigned long long) * nb, cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(hh.data() + nb, nsplit, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaMemcpyAsync(&n_active, d_active, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaGetLastError());
    PS_CUDA(cudaStreamSynchronize(st));
    int64_t npieces = 0, npieces_active = 0, m_active = 0;
    for (int k = 0; k < nb; ++k) {
        npieces += (int64_t)hh[k];
        if (k <= kPiece) npieces_active += (int64_t)hh[k], m_active += k * (int64_t)hh[k];  // bucket k: pieces of k edges
    }
    nv->settle();
    // publish the new version: queries that start from now on read it, those in flight keep the old one
    DeviceGraph &ng = nv->dg;
    ng = dg;
    ng.m = m2;
    ng.in_off = nv->in_off.as<int64_t>();
    ng.out_off = nv->out_off.as<int64_t>();
    ng.in_col = nv->in_col.as<int32_t>();
    ng.out_col = nv->out_col.as<int32_t>();
    ng.w = nv->w.as<float>();
    ng.rec = nv->rec.as<int4>();
    ng.n_pieces = npieces;
    ng.n_pieces_active = npieces_active;
    ng.m_active = m_active;
    ng.piece_v = nv->piece_v.as<int32_t>();
    ng.piece_beg = nv->piece_beg.as<int64_t>();
    ng.piece_len = nv->piece_len.as<int32_t>();
    ng.n_split = (int32_t)hh[nb];
    ng.split_v = nv->split_v.as<int32_t>();
    ng.n_active = n_active;
    nv->epoch = old->epoch + 1;
    g->publish(nv);
    if (applied) *applied = hm[2];
    return PROBESIM_OK;
}

extern "C" {

probesim_status probesim_insert_edges(probesim_graph *g, const int32_t *src, const int32_t *dst, int64_t k,
                                      int64_t *applied, void *stream) {
    return apply_updates(g, src, dst, k, true, applied, (cudaStream_t)stream);
}

probesim_status probesim_delete_edges(probesim_graph *g, const int32_t *src, const int32_t *dst, int64_t k,
                                      int64_t *applied, void *stream) {
    return apply_updates(g, src, dst, k, false, applied, (cudaStream_t)stream);
}

probesim_status probesim_num_walks(const probesim_graph *g, double eps, int64_t *n_r) {
    if (!g || !n_r) return fail(PROBESIM_E_INVALID, "null argument");
    if (!(eps > 0.0 && eps < 1.0)) return fail(PROBESIM_E_INVALID, "eps must lie in (0, 1)");
    *n_r = num_walks(g->cfg.c, eps, g->cfg.delta, g->n);
    return PROBESIM_OK;
}

probesim_status probesim_sample_walks(probesim_graph *g, const probesim_query *q, int32_t nq, int32_t *nodes,
                                      int32_t *lens, int64_t capacity, void *stream) {
    if (!g || !nodes || !lens) return fail(PROBESIM_E_INVALID, "null argument");
    PS_TRY(check_queries(g, q, nq, false, 0));
    std::lock_guard<std::mutex> lk(g->mu);
    const std::shared_ptr<StoreVersion> snap = g->current();
    g_last_error.clear();
    Workspace *ws = &g->ws0;
    cudaStream_t st = (cudaStream_t)stream;
    BatchPlan P;
    PS_TRY(plan_batch(g, q, nq, P));
    if (P.W > capacity) return fail(PROBESIM_E_INVALID, "walk buffer too small");
    QueryBatch qb;
    PS_TRY(upload_batch(ws, P, qb, st));
    const int32_t L = g->cfg.l_max;
    const bool dev_nodes = is_device_ptr(nodes), dev_lens = is_device_ptr(lens);
    PS_CUDA(ws->walks.ensure(sizeof(int32_t) * std::max<int64_t>(1, (int64_t)P.W * L)));
    PS_CUDA(ws->lens.ensure(sizeof(int32_t) * std::max<int32_t>(1, P.W)));
    PS_CUDA(ws->ctr.ensure(sizeof(LaunchCounters)));
    PS_CUDA(cudaMemsetAsync(ws->ctr.p, 0, sizeof(LaunchCounters), st));
    int32_t *wd = dev_nodes ? nodes : ws->walks.as<int32_t>();
    int32_t *ld = dev_lens ? lens : ws->lens.as<int32_t>();
    launch_walks(snap->dg, qb, P.W, L, g->t_stop, g->cfg.seed, wd, ld, true, ws->ctr.as<LaunchCounters>(), st);
    ps::launch_map_ids(wd, (int64_t)P.W * L, snap->dg.int2ext, st);
    PS_CUDA(cudaGetLastError());
    if (!dev_nodes)
        PS_CUDA(cudaMemcpyAsync(nodes, wd, sizeof(int32_t) * (size_t)P.W * L, cudaMemcpyDeviceToHost, st));
    if (!dev_lens) PS_CUDA(cudaMemcpyAsync(lens, ld, sizeof(int32_t) * (size_t)P.W, cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    return PROBESIM_OK;
}

}  // extern "C"

// Single-source estimates of nq queries into `scores` (host or device) using workspace ws.  The caller holds
// the store lock (shared) and owns ws.
probesim_status ps::single_source_core(probesim_graph *g, Workspace *ws, const std::shared_ptr<StoreVersion> &snap,
                                          const probesim_query *q, int32_t nq, float *scores, cudaStream_t st) {
    ws->stats = probesim_stats{};
    ws->snap = snap;
    ws->dg = snap->dg;
    struct Release {
        Workspace *w;
        ~Release() { w->snap.reset(); }
    } release{ws};
    const bool dev = is_device_ptr(scores);
    float *d_out = scores;
    const size_t out_bytes = sizeof(float) * (size_t)nq * g->n;
    if (!dev) {
        PS_CUDA(ws->out_stage.ensure(out_bytes));
        d_out = ws->out_stage.as<float>();
    }
    PS_TRY(run_queries(g, ws, q, nq, d_out, st));
    if (!dev) {
        PS_CUDA(cudaMemcpyAsync(scores, d_out, out_bytes, cudaMemcpyDeviceToHost, st));
        PS_CUDA(cudaStreamSynchronize(st));
    }
    return PROBESIM_OK;
}

// Top-k of nq queries (ids/vals host or device, [nq][kmax]) using workspace ws; same locking as above.
probesim_status ps::topk_core(probesim_graph *g, Workspace *ws, const std::shared_ptr<StoreVersion> &snap,
                                 const probesim_query *q, int32_t nq, int32_t kmax, int32_t *ids, float *vals,
                                 cudaStream_t st) {
    ws->stats = probesim_stats{};
    ws->snap = snap;
    ws->dg = snap->dg;
    struct Release {
        Workspace *w;
        ~Release() { w->snap.reset(); }
    } release{ws};
    const int32_t n = g->n;
    // scores of a chunk of queries, then the selection
    const int32_t chunk = (int32_t)std::max<int64_t>(1, std::min<int64_t>(nq, (int64_t)(budget_of(g, ws) / 8) / ((int64_t)n * 4)));
    PS_CUDA(ws->out_stage.ensure(sizeof(float) * (size_t)chunk * n));
    const int nblk = topk_blocks_per_query(n);
    PS_CUDA(ws->tk_hist.ensure(sizeof(unsigned) * 256 * chunk));
    PS_CUDA(ws->tk_state.ensure(sizeof(unsigned) * 4 * chunk));
    PS_CUDA(ws->tk_tie.ensure(sizeof(unsigned) * (size_t)nblk * chunk));
    PS_CUDA(ws->tk_cid.ensure(sizeof(int32_t) * (size_t)kmax * chunk));
    PS_CUDA(ws->tk_cval.ensure(sizeof(float) * (size_t)kmax * chunk));
    PS_CUDA(ws->tk_qk.ensure(sizeof(int32_t) * 2 * chunk));
    // the short way's candidate lists are as large as 8,192 scores a query: within the scores' share of the budget only
    const bool use_short = kmax <= kShortMaxK && topk_short_bytes(n, chunk) <= budget_of(g, ws) / 8;
    if (use_short) PS_CUDA(ws->tk_short.ensure(topk_short_bytes(n, chunk)));
    const bool dev_ids = is_device_ptr(ids), dev_vals = is_device_ptr(vals);
    // the lists of a chunk on the device: ids, scores, then the flag of the short way.  Short lists for host memory come
    // back in one copy through pinned memory (each pageable copy waits for the device, about 10 us)
    const size_t list = (size_t)kmax * chunk;
    const bool pinned = list <= ((size_t)1 << 20);
    const size_t pin_bytes = sizeof(int32_t) * std::max(pinned ? 2 * list + 1 : (size_t)1, 2 * (size_t)chunk);
    PS_CUDA(ws->tk_ids.ensure(sizeof(int32_t) * (2 * list + 1)));
    for (int32_t done = 0; done < nq; done += chunk) {
        const int32_t B = std::min(chunk, nq - done);
        PS_TRY(run_queries(g, ws, q + done, B, ws->out_stage.as<float>(), st));
        PS_CUDA(ws->pin_q.ensure(pin_bytes));
        int32_t *h = ws->pin_q.as<int32_t>();
        for (int32_t b = 0; b < B; ++b) {
            h[b] = q[done + b].node;
            h[B + b] = q[done + b].k;
        }
        int32_t *d_qn = ws->tk_qk.as<int32_t>(), *d_qk = d_qn + B;
        PS_CUDA(cudaMemcpyAsync(d_qn, h, sizeof(int32_t) * 2 * B, cudaMemcpyHostToDevice, st));
        TopkScratch sc;
        sc.hist = ws->tk_hist.as<unsigned>();
        sc.state = ws->tk_state.as<unsigned>();
        sc.tiecnt = ws->tk_tie.as<unsigned>();
        sc.cand_id = ws->tk_cid.as<int32_t>();
        sc.cand_val = ws->tk_cval.as<float>();
        const size_t LB = (size_t)B * kmax;
        int32_t *stage = ws->tk_ids.as<int32_t>(), *d_over = stage + 2 * LB;
        int32_t *oi = dev_ids ? ids + (int64_t)done * kmax : stage;
        float *ov = dev_vals ? vals + (int64_t)done * kmax : reinterpret_cast<float *>(stage + LB);
        // brings what belongs in host memory back, and the short way's flag
        auto finish = [&](bool flag) -> probesim_status {
            PS_CUDA(cudaGetLastError());
            const size_t from = !pinned ? 2 * LB : (!dev_ids ? 0 : (!dev_vals ? LB : 2 * LB)), to = 2 * LB + (flag ? 1 : 0);
            int32_t *hp = h + (pinned ? from : 0);
            if (to > from)
                PS_CUDA(cudaMemcpyAsync(hp, stage + from, sizeof(int32_t) * (to - from), cudaMemcpyDeviceToHost, st));
            if (!pinned && !dev_ids)
                PS_CUDA(cudaMemcpyAsync(ids + (int64_t)done * kmax, oi, sizeof(int32_t) * LB, cudaMemcpyDeviceToHost, st));
            if (!pinned && !dev_vals)
                PS_CUDA(cudaMemcpyAsync(vals + (int64_t)done * kmax, ov, sizeof(float) * LB, cudaMemcpyDeviceToHost, st));
            PS_CUDA(cudaStreamSynchronize(st));
            if (pinned && !dev_ids) std::memcpy(ids + (int64_t)done * kmax, h, sizeof(int32_t) * LB);
            if (pinned && !dev_vals) std::memcpy(vals + (int64_t)done * kmax, h + LB, sizeof(float) * LB);
            return PROBESIM_OK;
        };
        bool full = !use_short;
        if (use_short) {
            launch_topk_short(n, B, ws->out_stage.as<float>(), d_qn, d_qk, kmax, ws->tk_short.p, oi, ov, d_over, st,
                              &ws->stats.kernel_launches);
            PS_TRY(finish(true));
            full = h[pinned ? 2 * LB : 0] != 0;
        }
        if (full) {
            launch_topk(n, B, ws->out_stage.as<float>(), d_qn, d_qk, kmax, sc, oi, ov, st, &ws->stats.kernel_launches);
            PS_TRY(finish(false));
        }
    }
    return PROBESIM_OK;
}

extern "C" {

probesim_status probesim_single_source(probesim_graph *g, const probesim_query *q, int32_t nq, float *scores,
                                       void *stream) {
    if (!g || !scores) return fail(PROBESIM_E_INVALID, "null argument");
    PS_TRY(check_queries(g, q, nq, false, 0));
    std::lock_guard<std::mutex> lk(g->mu);
    g_last_error.clear();
    return single_source_core(g, &g->ws0, g->current(), q, nq, scores, (cudaStream_t)stream);
}

probesim_status probesim_topk(probesim_graph *g, const probesim_query *q, int32_t nq, int32_t kmax, int32_t *ids,
                              float *vals, void *stream) {
    if (!g || !ids || !vals) return fail(PROBESIM_E_INVALID, "null argument");
    if (kmax < 1 || kmax > 4096 || kmax > g->n - 1) return fail(PROBESIM_E_INVALID, "kmax must lie in [1, min(4096, n-1)]");
    PS_TRY(check_queries(g, q, nq, true, kmax));
    std::lock_guard<std::mutex> lk(g->mu);
    g_last_error.clear();
    return topk_core(g, &g->ws0, g->current(), q, nq, kmax, ids, vals, (cudaStream_t)stream);
}

// Times the pulls that the level loop launches below depth 0 (pull_full, pull_tail: the same kernels, chosen by the same
// rules, over the same pieces) for {2, 4, 8, 16} blocks per SM, keeps the fastest number for each kernel, and picks the
// full tiles' shape.  What is not faster than the default by more than kTunerGain stays at the default: a choice within
// the timings' noise must not make a tuned graph slower than an untuned one.  The choice is stored in the graph and used by
// every later query.  (Timing 32-column tiles alone over 64 columns, as this did, gave the wide tiles 2 blocks per SM: a
// query of two on 50,000 nodes and 5 million edges 8.4 ms untuned, 9.2 tuned; R-MAT 2^18 at eps 0.05 31.2 and 32.4.)
probesim_status probesim_autotune(probesim_graph *g, void *stream) {
    if (!g) return fail(PROBESIM_E_INVALID, "graph is null");
    std::lock_guard<std::mutex> lk(g->mu);
    const std::shared_ptr<StoreVersion> snap = g->current();
    g_last_error.clear();
    cudaStream_t st = (cudaStream_t)stream;
    DeviceGraph dg = snap->dg;
    dg.n_pieces = dg.n_pieces_active;
    if (dg.n_pieces == 0) return PROBESIM_OK;  // no edges: nothing is pulled below depth 0
    const int32_t n = dg.n, nt = tuner_tiles(n, dg.n_pieces, dg.n_active, budget_of(g, &g->ws0) / 2);
    const ColLayout L = make_layout(n, 32 * nt);
    Workspace *ws = &g->ws0;
    const size_t bytes = sizeof(float) * (size_t)L.size();
    PS_CUDA(ws->md_a.ensure(bytes));
    PS_CUDA(ws->md_b.ensure(bytes));
    PS_CUDA(cudaMemsetAsync(ws->md_a.p, 0x3c, bytes, st));  // any finite values
    PS_CUDA(cudaMemsetAsync(ws->md_b.p, 0, bytes, st));
    PS_CUDA(ws->pull_err.ensure(sizeof(int32_t)));
    PS_CUDA(cudaMemsetAsync(ws->pull_err.p, 0, sizeof(int32_t), st));
    const float *D = ws->md_a.as<float>();
    float *M = ws->md_b.as<float>();
    Timer tm{ws, st};
    const cudaEvent_t e0 = tm.get(), e1 = tm.get();
    PullTuning t = g->tune;
    int64_t launches = 0;
    cudaError_t le = cudaSuccess;
    // the shortest of three runs after a warm-up run, in ms
    auto time_pull = [&](auto &&launch) -> float {
        float best = 1e30f;
        for (int rep = 0; rep < 4; ++rep) {
            cudaEventRecord(e0, st);
            launch();
            cudaEventRecord(e1, st);
            if (cudaEventSynchronize(e1) != cudaSuccess) return 1e30f;
            float ms = 0.f;
            cudaEventElapsedTime(&ms, e0, e1);
            if (rep > 0) best = std::min(best, ms);
        }
        return best;
    };
    const float kTunerGain = 0.98f;
    // blocks per SM of one kernel, into `slot`; returns its time
    auto tune_blocks = [&](int32_t &slot, auto &&launch) -> float {
        int32_t pick = slot = kPullBlocks;
        float best = time_pull(launch);
        for (int32_t bps : {2, 4, 16}) {
            slot = bps;
            const float ms = time_pull(launch);
            if (ms < kTunerGain * best) best = ms, pick = bps;
        }
        slot = pick;
        return best;
    };
    // tail tiles: one narrow tile over a compact [n][T] block
    for (int32_t T : {1, 2, 4, 8, 16}) {
        const ColLayout LT = make_layout(n, T);
        tune_blocks(narrow_tail(dg.n_pieces) ? t.narrow[T] : t.bps[T],
                    [&] { pull_tail(dg, t, D, LT, M, LT, 0, T, nullptr, st); });
    }
    // full tiles, each shape over the same nt tiles: with 32 the wide tiles, and the 32-column ones left over or alone
    auto full = [&](int32_t tiles) {
        const cudaError_t e =
            pull_full(dg, t, D, L, M, L, tiles, nullptr, ws->pull_err.as<int32_t>(), &launches, st);
        if (e != cudaSuccess) le = e;
    };
    t.shape = 32;
    const FullTiles f = full_tiles(nt, dg.n_pieces, dg.n_active);
    float best = tune_blocks(t.bps[32], [&] { full(f.wide > 0 ? f.per - 1 : nt); });
    if (f.wide > 0) best = tune_blocks(t.bps[f.tile], [&] { full(nt); });
    const PullTuning base = t;
    PullTuning pick = t;
    for (int32_t shape : {16, kPullPairs, kPullTma}) {
        if (shape == kPullTma && !pull_tma_available()) continue;
        t = base;
        t.shape = shape;
        t.bps[kPullTma] = 1;  // the TMA launch: one block of 192 KB shared memory per SM
        const float ms = shape == kPullTma ? time_pull([&] { full(nt); }) : tune_blocks(t.bps[shape], [&] { full(nt); });
        if (ms < kTunerGain * best) best = ms, pick = t;
    }
    PS_CUDA(le);
    PS_CUDA(cudaGetLastError());
    int32_t herr = 0;
    PS_CUDA(cudaMemcpyAsync(&herr, ws->pull_err.p, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    PS_CUDA(cudaStreamSynchronize(st));
    if (herr) return fail(PROBESIM_E_TIMEOUT, "a TMA row gather of the pull did not complete in time");
    g->tune = pick;
    return PROBESIM_OK;
}

probesim_status probesim_set_tuning(probesim_graph *g, int32_t wide_tile, const int32_t *blocks_per_sm) {
    if (!g) return fail(PROBESIM_E_INVALID, "graph is null");
    if (wide_tile != 16 && wide_tile != 32 && wide_tile != kPullPairs && wide_tile != kPullTma)
        return fail(PROBESIM_E_INVALID, "wide_tile must be 16, 32, 64 or 96");
    if (wide_tile == kPullTma && !pull_tma_available())
        return fail(PROBESIM_E_UNSUPPORTED, "no tensor-map encoder in this driver");
    if (blocks_per_sm)
        for (int i = 0; i < 8; ++i)
            if (blocks_per_sm[i] < 1 || blocks_per_sm[i] > 32)
                return fail(PROBESIM_E_INVALID, "blocks_per_sm must lie in [1, 32]");
    std::lock_guard<std::mutex> lk(g->mu);
    g->tune.shape = wide_tile;
    if (blocks_per_sm) {
        for (int i = 0; i < 6; ++i) g->tune.bps[1 << i] = blocks_per_sm[i];
        for (int i = 0; i < 5; ++i) g->tune.narrow[1 << i] = blocks_per_sm[i];
        g->tune.bps[kPullWide] = g->tune.bps[kPullMid] = blocks_per_sm[5];
        g->tune.bps[kPullPairs] = blocks_per_sm[6];
        g->tune.bps[kPullTma] = blocks_per_sm[7];
    }
    return PROBESIM_OK;
}

probesim_status probesim_get_tuning(const probesim_graph *g, int32_t *wide_tile, int32_t *blocks_per_sm) {
    if (!g) return fail(PROBESIM_E_INVALID, "graph is null");
    const PullTuning &t = g->tune;
    if (wide_tile) *wide_tile = t.shape;
    if (blocks_per_sm) {  // of the kernels that pull below depth 0: the narrow tails, the wide tiles
        const std::shared_ptr<StoreVersion> v = const_cast<probesim_graph *>(g)->current();
        const bool narrow = narrow_tail(v->dg.n_pieces_active);
        const int32_t wide = v->dg.n_active <= kPullWideRows ? kPullWide : kPullMid;
        for (int i = 0; i < 6; ++i) {
            const int32_t b = i == 5 ? t.bps[wide] : (narrow ? t.narrow[1 << i] : t.bps[1 << i]);
            blocks_per_sm[i] = b ? b : kPullBlocks;
        }
    }
    return PROBESIM_OK;
}

probesim_status probesim_set_profiling(probesim_graph *g, int32_t on) {
    if (!g) return fail(PROBESIM_E_INVALID, "graph is null");
    std::lock_guard<std::mutex> lk(g->mu);
    g->ws0.profiling = on ? 1 : 0;
    return PROBESIM_OK;
}

probesim_status probesim_get_stats(const probesim_graph *g, probesim_stats *out) {
    if (!g || !out) return fail(PROBESIM_E_INVALID, "null argument");
    *out = g->ws0.stats;
    return PROBESIM_OK;
}

}  // extern "C"
