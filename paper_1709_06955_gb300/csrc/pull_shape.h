// Which kernel pulls the columns of a depth: the rules of the level loop, which the tuner times by the same rules.  Plain
// host code.
#pragma once

#include <algorithm>
#include <cstdint>

namespace ps {

// Launch shapes of the full 32-column tiles (probesim_set_tuning): 16-column halves (16), 32-column tiles (32), 32-column
// tiles two per pass, 32-column tiles whose rows the TMA gathers.
constexpr int32_t kPullPairs = 64;
constexpr int32_t kPullTma = 96;
// With 32: 128-column tiles (kPullWide) or 64-column ones (kPullMid).  The level loop takes full 32-column tiles four at a
// time the first way while the rows its gathers read (n_active of them) fit the L2 at 128 columns, else two at a time; and
// one at a time when the wide tiles would not fill the chip (a warp or half a warp per piece and tile: kPullWideWarps) --
// on a graph of 1,000 nodes they left most of it idle and cost a launch (1.02 -> 1.04 ms a query).
constexpr int32_t kPullWide = 128, kPullMid = 192;
constexpr int64_t kPullWideWarps = 2 * 152 * 32;
constexpr int64_t kPullWideRows = (128ll << 20) / 512;
// A depth's last 1 to 16 columns go to k_pull_narrow (pull_narrow.cu) on graphs of at most kNarrowPieces pieces: four
// times the threads the chip holds at eight lanes a piece (beyond that both kernels are bound by the gathers: 78 us
// against 82 for one column of R-MAT 2^20, where 22 against 5 on 30,000 nodes).
constexpr int64_t kNarrowPieces = 4ll * 152 * 2048 / 8;

// Blocks per SM of each pull kernel (0: the default) and the full tiles' shape.
constexpr int32_t kPullBlocks = 8;
struct PullTuning {
    int32_t shape = 32;
    int32_t bps[kPullMid + 1] = {0};  // k_pull by tile width, kPullPairs, kPullTma, kPullWide, kPullMid
    int32_t narrow[17] = {0};         // k_pull_narrow by tile width
};

// The full tiles of one depth with shape 32: `wide` launches' worth of `tile` (each `per` 32-column tiles), then `rest`
// 32-column tiles.
struct FullTiles {
    int32_t tile, per, wide, rest;
};
inline FullTiles full_tiles(int32_t nfull, int64_t n_pieces, int32_t n_active) {
    FullTiles f;
    f.per = n_active <= kPullWideRows ? 4 : 2;
    f.tile = f.per == 4 ? kPullWide : kPullMid;
    f.wide = nfull / f.per;
    if (n_pieces * f.wide * f.per / 4 < kPullWideWarps) f.wide = 0;
    f.rest = nfull - f.per * f.wide;
    return f;
}
inline bool narrow_tail(int64_t n_pieces) { return n_pieces <= kNarrowPieces; }

// 32-column tiles of the tuner's score matrix: four wide tiles, or as many as full_tiles wants before it takes wide ones
// (at most 4,096 columns), in at most 1 GB and `bytes` (two tiles however large the graph).
inline int32_t tuner_tiles(int32_t n, int64_t n_pieces, int32_t n_active, uint64_t bytes) {
    const int32_t per = n_active <= kPullWideRows ? 4 : 2;
    const int64_t fill = (4 * kPullWideWarps / per + std::max<int64_t>(1, n_pieces) - 1) / std::max<int64_t>(1, n_pieces);
    const int64_t want = std::min<int64_t>(128, per * std::max<int64_t>(4, fill));
    const int64_t room = (int64_t)std::min<uint64_t>(bytes, 1ull << 30) / (128 * ((int64_t)n + 1)) / per * per;
    return (int32_t)std::max<int64_t>(2, std::min(want, room));
}

}  // namespace ps
