// Pairwise Monte Carlo SimRank (Sec. 2.2, Eq. 3): s(u, v) is the probability that a sqrt(c)-walk from u and one
// from v meet, i.e. have the same i-th node for some i.  For r walk pairs the estimate is (pairs that meet) / r;
// with r >= ln(1/delta) / (2 eps^2) it is within eps of s(u, v) with probability 1 - delta (Chernoff).  It serves
// as the single-pair "expert" that gauges pooled top-k candidates on graphs too large for the Power Method.
//
// The two walks of a walk pair t advance in lockstep, their i-th nodes compared at every position both reach.  Walk t
// from u draws Philox counter (t, s, 0, 0) under key (seed, key_u) at step s -- the draws of query key_u's walk t in the
// single-source path -- and likewise from v under (seed, key_v).
#include <algorithm>

#include "internal.cuh"

namespace ps {

namespace {

constexpr int kThreads = 256;

// grid.y = pair; meets[pair] += walk pairs t in [0, r) that meet.  A thread takes its next walk pair as soon as one ends
// (both walks go on with probability c, so a pair takes 2.5 steps on average, the longest of a warp's 32 about 8): the
// loop's body is one step of whatever pair the thread holds.  A step's draws come before its gathers, which only pairs
// that go on make: the node records of both nodes, then one in-list entry each.
// What bounds it: issue slots (68 % of the SM busy, two thirds of it Philox).  50 pairs of 2^20 walk pairs on R-MAT
// 2^20: 1.51 ms with a loop over pairs around a loop over steps, 0.59 now (0.79 with 8 blocks per SM, 0.65 with 128).
__global__ void __launch_bounds__(kThreads) k_pair_mc(const int4 *__restrict__ rec, const int32_t *__restrict__ in_col,
                                                      const int32_t *__restrict__ ext2int, const int32_t *__restrict__ pu,
                                                      const int32_t *__restrict__ pv, const uint32_t *__restrict__ ku,
                                                      const uint32_t *__restrict__ kv, int64_t r, int32_t l_max,
                                                      uint32_t seed, uint32_t t_stop,
                                                      unsigned long long *__restrict__ meets) {
    __shared__ unsigned s_cnt;
    if (threadIdx.x == 0) s_cnt = 0;
    __syncthreads();
    const int32_t pair = blockIdx.y;
    const int32_t u0 = ext2int[pu[pair]], v0 = ext2int[pv[pair]];
    const uint32_t keyu = ku[pair], keyv = kv[pair];
    const int4 ru = rec[u0], rv = rec[v0];
    const int64_t step = (int64_t)gridDim.x * blockDim.x;
    unsigned local = 0;
    int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (u0 == v0) {  // equal nodes meet at once
        for (; t < r; t += step) ++local;
    } else {
        int32_t a = u0, b = v0;
        int4 ra = ru, rb = rv;
        uint32_t s = 0;
        while (t < r) {
            // positions 1, 2, ... exist while both walks continue; a walk holds at most l_max nodes
            const U32x4 da = philox4x32_10((uint32_t)t, s, 0u, 0u, seed, keyu);
            const U32x4 db = philox4x32_10((uint32_t)t, s, 0u, 0u, seed, keyv);
            bool on = da.x >= t_stop && db.x >= t_stop && (int32_t)s + 1 < l_max;
            if (on && s > 0) {
                ra = __ldg(rec + a);
                rb = __ldg(rec + b);
            }
            on = on && ra.y > 0 && rb.y > 0;
            bool meet = false;
            if (on) {
                a = __ldg(in_col + ra.x + (int32_t)__umulhi(da.y, (uint32_t)ra.y));
                b = __ldg(in_col + rb.x + (int32_t)__umulhi(db.y, (uint32_t)rb.y));
                meet = a == b;
                ++s;
            }
            if (!on || meet) {  // the next pair, from the start
                local += meet;
                t += step;
                s = 0;
                ra = ru;
                rb = rv;
            }
        }
    }
    for (int o = 16; o; o >>= 1) local += __shfl_xor_sync(0xffffffffu, local, o);
    if ((threadIdx.x & 31) == 0 && local) atomicAdd(&s_cnt, local);
    __syncthreads();
    if (threadIdx.x == 0 && s_cnt) atomicAdd(meets + pair, (unsigned long long)s_cnt);
}

}  // namespace

void launch_pair_mc(const DeviceGraph &g, const int32_t *pu, const int32_t *pv, const uint32_t *ku, const uint32_t *kv,
                    int32_t npairs, int64_t r, int32_t l_max, uint32_t seed, uint32_t t_stop, unsigned long long *meets,
                    cudaStream_t s) {
    if (npairs <= 0 || r <= 0) return;
    int dev = 0, sms = 152;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    int64_t bx = (r + kThreads - 1) / kThreads;  // blocks per pair: about 32 per SM over all pairs
    bx = std::min<int64_t>(bx, std::max<int64_t>(1, (int64_t)sms * 32 / npairs));
    dim3 grid((unsigned)bx, (unsigned)npairs);
    k_pair_mc<<<grid, kThreads, 0, s>>>(g.rec, g.in_col, g.ext2int, pu, pv, ku, kv, r, l_max, seed, t_stop, meets);
}

}  // namespace ps
