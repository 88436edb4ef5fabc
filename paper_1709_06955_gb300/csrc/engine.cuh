// Host-side engine types shared by the C ABI (probesim.cu) and the serving loop (server.cu).
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <memory>
#include <mutex>
#include <string>
#include <vector>

#include "buffers.h"
#include "internal.cuh"
#include "level_plan.h"
#include "rand_lists.h"

// One version of the graph store.  A query holds the version it started with; an update batch builds the next
// version beside it and publishes it, so queries never wait for updates nor updates for queries, and a version's
// device memory is freed when its last reader lets go.
struct StoreVersion {
    DevBuf arena;  // the first version: one allocation that the arrays below are parts of
    DevBuf in_off, in_col, out_off, out_col, w, rec, piece_v, piece_beg, piece_len, split_v;
    std::shared_ptr<StoreVersion> base;  // set when this version reuses base's arrays (an update that changed nothing)
    ps::DeviceGraph dg;
    uint64_t epoch = 0;
    void settle() {  // every array is written
        for (DevBuf *b : {&in_off, &in_col, &out_off, &out_col, &w, &rec, &piece_v, &piece_beg, &piece_len, &split_v})
            b->settle();
    }
    ~StoreVersion() {
        for (DevBuf *b : {&in_off, &in_col, &out_off, &out_col, &w, &rec, &piece_v, &piece_beg, &piece_len, &split_v, &arena})
            b->release();
    }
};

// Per-call device and pinned buffers; a graph owns one for direct calls, a server one per worker.
struct Workspace {
    DevBuf qbuf, walks, lens, ctr;
    DevBuf t_key, t_node, t_parent, t_depth, t_query, t_weight, t_height, t_slot, t_gamma, t_G;
    DevBuf counts, node_list, sched;  // level schedule: node counts and lists per depth, uploaded plan
    ps::LevelPlan plan;               // its host side
    DevBuf md_a, md_b, out_stage;     // the two score buffers; host-output staging
    DevBuf r_ent[2], r_first[2], r_counts, r_counts2, r_ctr;
    DevBuf tk_hist, tk_state, tk_tie, tk_cid, tk_cval, tk_ids, tk_qk, tk_short;
    // frontier engine: walk-prefix slots, switched flags, probes, frontier lists, deferral stack, tasks, global tables,
    // estimates
    DevBuf f_wslot, f_tsw, f_slot, f_misc, f_pr32, f_pr64, f_acc, f_tab, f_list[2], f_stack, f_tasks, f_keys;
    DevBuf pm_in, pm_meets;  // pairwise Monte Carlo: pairs and keys, meet counts
    DevBuf pull_err;         // set by the TMA pull when a stage's wait gives up
    bool f_table_clean = false;  // f_keys (the global tables) holds only empty slots (every sweep empties its slots)
    PinnedBuf pin_q;  // query arrays of one batch; exported tree nodes; the plan on its way up
    PinnedBuf pin_s;  // counters and schedule offsets (fixed size, allocated at creation)
    int profiling = 0;
    size_t budget = 0;  // device memory one call on this workspace may take; 0 = the graph's budget
    std::shared_ptr<StoreVersion> snap;  // the store version of the call in progress
    ps::DeviceGraph dg;                  // its device view
    std::vector<cudaEvent_t> ev;
    probesim_stats stats{};
    // a second stream for work of a depth that runs beside the pull (the push block, the tail tile), and the
    // events that order it against the caller's stream; created on first use
    cudaStream_t side = nullptr;
    cudaEvent_t ev_start = nullptr, ev_ready = nullptr, ev_side = nullptr;
    cudaError_t ensure_side() {
        if (side) return cudaSuccess;
        cudaError_t e = cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_start, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_ready, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_side, cudaEventDisableTiming);
        return e;
    }
    void release() {
        DevBuf *bufs[] = {&qbuf, &walks, &lens, &ctr, &t_key, &t_node, &t_parent, &t_depth, &t_query, &t_weight,
                          &t_height, &t_slot, &t_gamma, &t_G, &counts, &node_list,
                          &sched, &md_a, &md_b, &out_stage, &r_ent[0], &r_ent[1], &r_first[0], &r_first[1],
                          &r_counts, &r_counts2, &r_ctr, &tk_hist, &tk_state, &tk_tie,
                          &tk_cid, &tk_cval, &tk_ids, &tk_qk, &tk_short, &f_wslot, &f_tsw, &f_slot, &f_misc, &f_pr32, &f_pr64, &f_acc,
                          &f_tab, &f_list[0], &f_list[1], &f_stack, &f_tasks, &f_keys, &pm_in, &pm_meets, &pull_err};
        for (DevBuf *b : bufs) b->release();
        f_table_clean = false;
        pin_q.release();
        pin_s.release();
        for (cudaEvent_t e : ev) cudaEventDestroy(e);
        ev.clear();
        for (cudaEvent_t *e : {&ev_start, &ev_ready, &ev_side})
            if (*e) cudaEventDestroy(*e), *e = nullptr;
        if (side) cudaStreamDestroy(side), side = nullptr;
    }
};

struct probesim_graph {
    std::mutex mu;              // serialises direct calls (they share ws0)
    std::mutex update_mu;       // serialises update batches
    std::mutex store_ptr_mu;    // guards the pointer to the current store version
    std::shared_ptr<StoreVersion> store;
    probesim_config cfg{};
    uint32_t t_stop = 0;
    uint32_t t_keep = 0;
    int device = 0;
    int32_t n = 0;              // node count (fixed; updates change edges only)
    DevBuf ext2int, int2ext;    // the id maps, shared by every store version
    std::shared_ptr<StoreVersion> current() {
        std::lock_guard<std::mutex> lk(store_ptr_mu);
        return store;
    }
    void publish(std::shared_ptr<StoreVersion> v) {
        std::lock_guard<std::mutex> lk(store_ptr_mu);
        store.swap(v);  // the old version is released outside the lock, by whichever reader holds it last
    }
    // update scratch
    DevBuf u_batch, u_valid, u_vpre, u_delta, u_deg, u_part, u_hist, u_bounds, u_raw, u_keys[3], u_sort;
    // update batches run on a stream of their own (under update_mu), created on first use
    cudaStream_t u_stream = nullptr;
    cudaEvent_t u_ready = nullptr;
    cudaError_t ensure_update_stream() {
        if (u_stream) return cudaSuccess;
        int low = 0, high = 0;
        cudaError_t e = cudaDeviceGetStreamPriorityRange(&low, &high);
        if (e == cudaSuccess && !u_ready) e = cudaEventCreateWithFlags(&u_ready, cudaEventDisableTiming);
        if (e == cudaSuccess) e = cudaStreamCreateWithPriority(&u_stream, cudaStreamNonBlocking, high);
        if (e != cudaSuccess) u_stream = nullptr;
        return e;
    }
    uint64_t epoch = 0;
    Workspace ws0;
    std::atomic<size_t> budget{0};  // device memory one call's working buffers may take (set while calls run)
    size_t budget0 = 0;  // the default: 60% of device memory at creation
    ps::PullTuning tune;  // the pull's launch shape: probesim_autotune, probesim_set_tuning (defaults until then)
};


namespace ps {
// Status helpers (probesim.cu): set the calling thread's message and return the status.
probesim_status fail_status(probesim_status st, const std::string &msg);
// Checks a query array against the graph (ids, eps, k <= kmax when topk).
probesim_status check_queries(const probesim_graph *g, const probesim_query *q, int32_t nq, bool topk, int32_t kmax);
// Estimates and top-k of nq queries with workspace ws on stream st, over store version snap.  The caller owns ws.
probesim_status single_source_core(probesim_graph *g, Workspace *ws, const std::shared_ptr<StoreVersion> &snap,
                                   const probesim_query *q, int32_t nq, float *scores, cudaStream_t st);
probesim_status topk_core(probesim_graph *g, Workspace *ws, const std::shared_ptr<StoreVersion> &snap,
                          const probesim_query *q, int32_t nq, int32_t kmax, int32_t *ids, float *vals, cudaStream_t st);
// Applies one update batch: builds the next store version from the current one and publishes it (serialised with
// other update batches, never waiting for queries).
probesim_status apply_updates(probesim_graph *g, const int32_t *src, const int32_t *dst, int64_t k, bool insert,
                              int64_t *applied, cudaStream_t st);
int64_t num_walks_for(const probesim_graph *g, double eps);
}  // namespace ps
