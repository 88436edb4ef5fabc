// The level loop's schedule: which column of a depth's score matrix each tree node owns, and what the accumulate adds
// where.  Plain host code; the device waits for it, so every step is linear in the column nodes: nodes are renumbered in
// entry order by a rank over a bitmap of the table (which also finds a node's parent), lists per depth and per parent are
// flat arrays filled by counting, and a chain's column comes from a bitmap of the columns given back.  (R-MAT 2^20, one
// query, 4,535 column nodes: 0.12 ms; with sorts, a segment tree over the columns and a vector of children per node it
// took 0.37.  R-MAT 2^18, two queries at eps 0.05, 32,376 nodes: 3.25 -> 0.95 ms.)
#pragma once

#include <algorithm>
#include <cstdint>
#include <vector>

namespace ps {

// A set of small integers that gives its smallest member: 64-ary bitmaps, a bit of a level above per word below.
struct SmallestFirst {
    std::vector<uint64_t> level[4];  // 64^4 members at most
    int levels = 0;
    void reset(int32_t n) {
        levels = 0;
        int64_t words = n;
        do {
            words = std::max<int64_t>(1, (words + 63) / 64);
            level[levels++].assign((size_t)words, 0);
        } while (words > 1 && levels < 4);
    }
    void insert(int32_t x) {
        for (int l = 0; l < levels; ++l, x >>= 6) level[l][x >> 6] |= 1ull << (x & 63);
    }
    int32_t take() {  // -1: empty
        int32_t w = -1;
        for (size_t i = 0; i < level[levels - 1].size() && w < 0; ++i)
            if (level[levels - 1][i]) w = (int32_t)i;
        if (w < 0) return -1;
        for (int l = levels - 1;; --l) {
            w = 64 * w + __builtin_ctzll(level[l][w]);
            if (l == 0) break;
        }
        int32_t x = w;
        for (int l = 0; l < levels; ++l, x >>= 6) {
            level[l][x >> 6] &= ~(1ull << (x & 63));
            if (level[l][x >> 6]) break;
        }
        return w;
    }
};

struct LevelPlan {
    // per depth: columns of the dense nodes, full 32-column tiles and the tail tile that cover them (dw columns in all),
    // push nodes in inherited columns, first column of the push block, columns in all
    std::vector<int32_t> width, nfull, tail, dw, hinh, h0, cols;
    std::vector<int32_t> rho;         // per query: its super-root's column, -1 without one
    std::vector<int32_t> ent, col;    // per column node, in entry order: its table entry and its column
    std::vector<int32_t> zmask, zoff, zany;  // the pull's zero masks (see below)
    // accumulate parts of depth d: first parts [p1_at[d], p1_at[d + 1]), later parts likewise; sources of the depth
    std::vector<int32_t> p1dst, p1src, p2dst, p2src, p1_at, p2_at;
    std::vector<int64_t> acc_src;

    // entry, parent, tag: per exported node (any order) its table entry, its parent's entry (-1 - query at depth 0) and
    // 2 * depth + (1 if dense).  cap: table slots; depths 0 .. D1 - 1; tile_for(r): the tail tile of r columns.
    // False if a node's parent was not exported.
    template <class TileFor>
    bool build(int32_t N, const int32_t *entry, const int32_t *parent, const int32_t *tag, int64_t cap, int32_t B,
               int32_t D1, TileFor tile_for) {
        // nodes in entry order
        bits.assign((size_t)(cap + 63) / 64, 0);
        for (int32_t i = 0; i < N; ++i) bits[entry[i] >> 6] |= 1ull << (entry[i] & 63);
        below.resize(bits.size());
        int32_t sum = 0;
        for (size_t w = 0; w < bits.size(); ++w) below[w] = sum, sum += __builtin_popcountll(bits[w]);
        auto rank = [&](int32_t e) {
            return below[e >> 6] + __builtin_popcountll(bits[e >> 6] & ((1ull << (e & 63)) - 1));
        };
        for (auto *v : {&ent, &par, &dep, &col}) v->resize(N);
        dense.resize(N);
        dn_at.assign(D1 + 1, 0);
        pn_at.assign(D1 + 1, 0);
        for (int32_t i = 0; i < N; ++i) {
            const int32_t r = rank(entry[i]), p = parent[i], d = tag[i] >> 1;
            if (d > 0 && (p < 0 || !(bits[p >> 6] >> (p & 63) & 1))) return false;
            ent[r] = entry[i];
            par[r] = d > 0 ? rank(p) : p;
            dep[r] = d;
            dense[r] = tag[i] & 1;
            ++(dense[r] ? dn_at : pn_at)[d + 1];
        }
        for (int32_t d = 0; d < D1; ++d) dn_at[d + 1] += dn_at[d], pn_at[d + 1] += pn_at[d];
        // dense and push nodes by depth, in entry order
        dl.resize(dn_at[D1]);
        pl.resize(pn_at[D1]);
        cur = dn_at;
        cur2 = pn_at;
        for (int32_t r = 0; r < N; ++r)
            if (dense[r]) dl[cur[dep[r]]++] = r;
            else pl[cur2[dep[r]]++] = r;
        // the heir of a node is its dense child with the deepest chain of dense descendants, ties to the smaller entry
        heir.assign(N, -1);
        chain.assign(N, 0);
        inherits.assign(N, 0);
        for (int32_t d = D1 - 1; d >= 1; --d)
            for (int32_t k = dn_at[d]; k < dn_at[d + 1]; ++k) {
                const int32_t i = dl[k], p = par[i];
                if (heir[p] < 0 || chain[i] > chain[heir[p]]) heir[p] = i;
                chain[p] = std::max(chain[p], chain[i] + 1);
            }
        // a dense node without one takes its first push child (smallest entry): that child's pushed column is then the
        // node's D column, in place, and the accumulate has nothing to copy
        hinh.assign(D1, 0);
        for (int32_t d = 1; d < D1; ++d)
            for (int32_t k = pn_at[d]; k < pn_at[d + 1]; ++k)
                if (heir[par[pl[k]]] < 0) {
                    heir[par[pl[k]]] = pl[k];
                    ++hinh[d];
                }
        for (int32_t i = 0; i < N; ++i)
            if (heir[i] >= 0) inherits[heir[i]] = 1;
        // A chain is a maximal path of heirs; its nodes share one column.  Chains are coloured deepest bottom first
        // (then by top, then by entry), each taking the smallest column whose chains all start more than one depth
        // below its bottom: a column whose chain ends at depth d stays unused at depth d + 1 too, where the accumulate
        // sets it while other groups may still read what a chain starting at d + 1 left in it.  Bottoms only rise, so a
        // column given back stays free until it is taken.
        head.clear();
        bottom.clear();
        cur.assign(D1 + 1, 0);
        for (int32_t x : dl) {
            if (inherits[x]) continue;
            head.push_back(x);
            int32_t b = dep[x];
            for (int32_t y = heir[x]; y >= 0; y = heir[y]) ++b;
            bottom.push_back(b);
            ++cur[b];
        }
        const int32_t chains = (int32_t)head.size();
        for (int32_t d = D1 - 1, at = 0; d >= 0; --d) {
            const int32_t c = cur[d];
            cur[d] = at;
            at += c;
        }
        order.resize(chains);
        for (int32_t k = 0; k < chains; ++k) order[cur[bottom[k]]++] = k;
        given.assign(D1 + 1, -1);  // columns by the top of their last chain, linked
        next.resize(chains);
        free_cols.reset(chains);
        int32_t opened = 0, seen = D1;  // tops >= seen are free
        for (int32_t k : order) {
            for (; seen > bottom[k] + 2; --seen)
                for (int32_t c = given[seen - 1]; c >= 0; c = next[c]) free_cols.insert(c);
            int32_t c = free_cols.take();
            if (c < 0) c = opened++;
            const int32_t top = dep[head[k]];
            next[c] = given[top];
            given[top] = c;
            for (int32_t x = head[k]; x >= 0; x = heir[x]) col[x] = c;
        }
        // columns and tiles of each depth: full 32-column tiles and one narrower tail tile of 1..16 columns
        for (auto *v : {&width, &nfull, &tail, &dw, &h0, &cols}) v->assign(D1, 0);
        rho.assign(B, -1);
        for (int32_t d = 0; d < D1; ++d) {
            for (int32_t k = dn_at[d]; k < dn_at[d + 1]; ++k) width[d] = std::max(width[d], col[dl[k]] + 1);
            int32_t full = width[d] / 32, rem = width[d] - 32 * full;
            if (rem > 16) ++full, rem = 0;
            nfull[d] = full;
            tail[d] = rem > 0 ? tile_for(rem) : 0;
            dw[d] = 32 * full + tail[d];
        }
        for (int32_t k = dn_at[0]; k < dn_at[1]; ++k) rho[-1 - par[dl[k]]] = col[dl[k]];
        // dense nodes of a depth in column order
        for (int32_t d = 0; d < D1; ++d) {
            at_col.assign(width[d], -1);
            for (int32_t k = dn_at[d]; k < dn_at[d + 1]; ++k) at_col[col[dl[k]]] = dl[k];
            int32_t k = dn_at[d];
            for (int32_t x : at_col)
                if (x >= 0) dl[k++] = x;
        }
        // the children that a node's accumulate reads, in column order: dense ones, then push ones
        kid_at.assign(N + 1, 0);
        for (int32_t i = 0; i < N; ++i)
            if (par[i] >= 0 && !inherits[i]) ++kid_at[par[i] + 1];
        for (int32_t i = 0; i < N; ++i) kid_at[i + 1] += kid_at[i];
        kid.resize(kid_at[N]);
        cur.assign(kid_at.begin(), kid_at.end() - 1);
        for (auto *l : {&dl, &pl})
            for (int32_t x : *l)
                if (par[x] >= 0 && !inherits[x]) kid[cur[par[x]]++] = x;
        // MD of depth d is read in place as D of depth d - 1, so its matrix holds the columns of both depths:
        // max(dw[d - 1], dw[d]) dense columns (inherited push columns among them), then the push block at h0[d], grouped
        // by parent in parent column order
        acc_src.assign(D1, 0);
        p1_at.assign(D1 + 1, 0);
        p2_at.assign(D1 + 1, 0);
        for (auto *v : {&p1dst, &p1src, &p2dst, &p2src}) v->clear();
        for (int32_t d = 0; d < D1; ++d) {
            const int32_t dense_w = std::max(dw[d], d >= 1 ? dw[d - 1] : 0);
            h0[d] = (std::max(dense_w, 1) + 3) / 4 * 4;
            cols[d] = (h0[d] + (pn_at[d + 1] - pn_at[d] - hinh[d]) + 3) / 4 * 4;
        }
        for (int32_t d = 0; d < D1; ++d) {
            p1_at[d] = (int32_t)p1dst.size();
            p2_at[d] = (int32_t)p2dst.size();
            int32_t push_col = d + 1 < D1 ? h0[d + 1] : 0;
            for (int32_t k = dn_at[d]; k < dn_at[d + 1]; ++k) {
                const int32_t i = dl[k], k0 = kid_at[i], k1 = kid_at[i + 1];
                for (int32_t j = k0; j < k1; ++j) {
                    const int32_t x = kid[j];
                    if (!dense[x]) col[x] = push_col++;
                    kid[j] = col[x];
                }
                // A group (the sum of the children's columns, into the parent's) is cut into parts of at most four
                // sources: a destination (bit 30: set, for a node without heir) and an int4 of sources (-1 = none).  The
                // first part of every group runs in the accumulate's first phase, the others add in a second phase (so
                // one node with many children does not hold up a block).
                const bool own = heir[i] < 0;
                if (k0 == k1 && !own) continue;  // its column already is its heir's MD
                acc_src[d] += k1 - k0;
                put_part(p1dst, p1src, col[i] | (own ? (1 << 30) : 0), k0, k1);
                for (int32_t f = k0 + 4; f < k1; f += 4) put_part(p2dst, p2src, col[i], f, k1);
            }
        }
        p1_at[D1] = (int32_t)p1dst.size();
        p2_at[D1] = (int32_t)p2dst.size();
        // zero masks of the pull at each depth: an inherited push column inside the pulled tiles is written as 0 there
        // (the push fills it afterwards); one 32-bit word per 32 columns, words of depth d at zoff[d]
        zoff.assign(D1 + 1, 0);
        zany.assign(D1, 0);
        for (int32_t d = 0; d < D1; ++d) zoff[d + 1] = zoff[d] + (dw[d] + 31) / 32;
        zmask.assign(zoff[D1], 0);
        for (int32_t x : pl) {
            const int32_t d = dep[x], c = col[x];
            if (inherits[x] && c < dw[d]) {
                zmask[zoff[d] + c / 32] |= (int32_t)(1u << (c % 32));
                zany[d] = 1;
            }
        }
        return true;
    }

private:
    std::vector<uint64_t> bits;
    std::vector<int32_t> below, par, dep, dn_at, pn_at, dl, pl, cur, cur2, heir, chain, head, bottom, order, given, next,
        at_col, kid_at, kid;
    std::vector<uint8_t> dense, inherits;
    SmallestFirst free_cols;

    void put_part(std::vector<int32_t> &dst, std::vector<int32_t> &src, int32_t dcol, int32_t from, int32_t end) {
        dst.push_back(dcol);
        for (int32_t j = from; j < from + 4; ++j) src.push_back(j < end ? kid[j] : -1);
    }
};

}  // namespace ps
