// The pull over one narrow tile (T = 1, 2, 4, 8 or 16 columns): MD[v][c] = sqrt(c)/|I(v)| * sum_{x in I(v)} D[x][c].
//
// Most depths of a walk tree are a few chains wide, so a call pulls a handful of columns many times in a row, each over
// the whole graph.  On a graph that does not fill the chip with a thread (or two, or four) per in-list piece, such a pull
// waits for the longest chain of gathers: a thread takes a piece's entries eight at a time.  Here eight lanes share a
// piece and take consecutive entries (T / 4 lanes an entry for T > 4), so a piece of 128 entries is 8 rounds of two
// loads, the indices of eight entries are one sector's lookup, and no lane needs another's index; the lanes' partial
// sums meet at the end of the piece.
// One column of a graph of 30,000 nodes and 400,000 edges: 22 us with a thread per piece, 5 with eight lanes; sixteen
// columns 12.4 and 9.6.
#include "internal.cuh"

namespace ps {

namespace {

// plain loads: the kernel ahead, which may still run when this one starts, writes what is gathered, so the read-only
// path is not for it
template <int VEC>
struct Vec {
    float a[VEC];
    __device__ __forceinline__ void load(const float *p) {
        if (VEC == 4) {
            const float4 v = *reinterpret_cast<const float4 *>(p);
            a[0] = v.x, a[1 % VEC] = v.y, a[2 % VEC] = v.z, a[3 % VEC] = v.w;
        } else if (VEC == 2) {
            const float2 v = *reinterpret_cast<const float2 *>(p);
            a[0] = v.x, a[1 % VEC] = v.y;
        } else {
            a[0] = *p;
        }
    }
};

// U steps of 8 lanes in flight
template <int T, int U>
__global__ void __launch_bounds__(256) k_pull_narrow(const int32_t *__restrict__ piece_v,
                                                     const int64_t *__restrict__ piece_beg,
                                                     const int32_t *__restrict__ piece_len, int64_t n_pieces,
                                                     const int32_t *__restrict__ in_col, const float *__restrict__ w,
                                                     const float *D, int32_t dpitch, float *MD,
                                                     int32_t pitch, int32_t zrow, const uint32_t *__restrict__ zmask) {
    pdl_wait();
    constexpr int VEC = T >= 4 ? 4 : T, LPE = T > 4 ? T / 4 : 1, EPS = 8 / LPE;  // lanes an entry, entries a step
    const int lane = threadIdx.x & 31, lig = lane & 7, sub = lig % LPE, slot = lig / LPE;
    const unsigned gmask = 0xffu << (lane - lig);
    uint32_t zbits = 0;  // this lane's columns that are written as 0 (the push fills them later)
    if (zmask != nullptr) zbits = (__ldg(zmask) >> (sub * VEC)) & ((1u << VEC) - 1u);
    const float *d0 = D + sub * VEC;
    const int64_t gid = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 3;
    const int64_t ngroups = ((int64_t)gridDim.x * blockDim.x) >> 3;
    auto load_meta = [&](int64_t q, int32_t &v, int64_t &beg, int32_t &info) {
        v = 0, beg = 0, info = 0;
        if (q < n_pieces) {
            v = __ldg(piece_v + q);
            beg = __ldg(piece_beg + q);
            info = __ldg(piece_len + q);
        }
    };
    auto load_idx = [&](int64_t beg, int32_t len, int32_t e0, int32_t (&x)[U]) {
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int32_t e = e0 + u * EPS + slot;
            x[u] = e < len ? __ldg(in_col + beg + e) : zrow;  // past the end: the zero spare row
        }
    };
    // the record of the piece after next and the next indices are loaded under the gathers
    int64_t p = gid, beg, beg1;
    int32_t v, info, v1, info1, x[U];
    load_meta(p, v, beg, info);
    load_meta(p + ngroups, v1, beg1, info1);
    load_idx(beg, info & 0x7fffffff, 0, x);
    for (; p < n_pieces; p += ngroups) {
        int32_t v2, info2;
        int64_t beg2;
        load_meta(p + 2 * ngroups, v2, beg2, info2);
        const float wv = __ldg(w + v);
        const int32_t len = info & 0x7fffffff;
        float acc[VEC];
#pragma unroll
        for (int k = 0; k < VEC; ++k) acc[k] = 0.f;
        for (int32_t e0 = 0;;) {
            Vec<VEC> val[U];
            if (len > 0) {
#pragma unroll
                for (int u = 0; u < U; ++u) val[u].load(d0 + (int64_t)x[u] * dpitch);
            }
            e0 += U * EPS;
            const bool more = e0 < len;
            if (more) load_idx(beg, len, e0, x);
            else load_idx(beg1, info1 & 0x7fffffff, 0, x);
            if (len > 0) {
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int k = 0; k < VEC; ++k) acc[k] += val[u].a[k];
            }
            if (!more) break;
        }
#pragma unroll
        for (int o = LPE; o < 8; o <<= 1)
#pragma unroll
            for (int k = 0; k < VEC; ++k) acc[k] += __shfl_xor_sync(gmask, acc[k], o);
        if (slot == 0) {
            float *dst = MD + (int64_t)v * pitch + sub * VEC;
#pragma unroll
            for (int k = 0; k < VEC; ++k) acc[k] = (zbits >> k) & 1u ? 0.f : acc[k] * wv;
            if (info < 0) {  // a piece of a cut in-list
#pragma unroll
                for (int k = 0; k < VEC; ++k) atomicAdd(dst + k, acc[k]);
            } else if (VEC == 4) {
                *reinterpret_cast<float4 *>(dst) = make_float4(acc[0], acc[1 % VEC], acc[2 % VEC], acc[3 % VEC]);
            } else if (VEC == 2) {
                *reinterpret_cast<float2 *>(dst) = make_float2(acc[0], acc[1 % VEC]);
            } else {
                dst[0] = acc[0];
            }
        }
        v = v1, beg = beg1, info = info1;
        v1 = v2, beg1 = beg2, info1 = info2;
    }
}

}  // namespace

void launch_pull_narrow(const DeviceGraph &g, const float *D, int32_t dpitch, float *MD, int32_t pitch, int32_t tile,
                        int32_t blocks_per_sm, const uint32_t *zmask, cudaStream_t s) {
    const int blocks = grid_for(g.n_pieces * 8, 256, blocks_per_sm > 0 ? blocks_per_sm : kPullBlocks);
#define PS_NARROW(T, U)                                                                                               \
    pdl_launch(k_pull_narrow<T, U>, dim3(blocks), dim3(256), 0, s, g.piece_v, g.piece_beg, g.piece_len, g.n_pieces,   \
               g.in_col, g.w, D, dpitch, MD, pitch, g.n, zmask)
    switch (tile) {
        case 1: PS_NARROW(1, 2); break;
        case 2: PS_NARROW(2, 2); break;
        case 4: PS_NARROW(4, 2); break;
        case 8: PS_NARROW(8, 4); break;
        default: PS_NARROW(16, 4); break;
    }
#undef PS_NARROW
}

}  // namespace ps
