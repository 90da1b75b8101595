// xd_window.h -- the tables of the window product (xd_u1_win.cu) on a large
// U(1) block: which bonds are done in which pass, and for every pass the
// words of its window, the flips between them and the tiles.  Plain C++
// without CUDA (the kernels read these tables; the CPU tests compile this
// header alone).
//
// A pass takes the bonds whose two sites lie in a window S of at most 12
// sites.  A word splits into its window word w (the bits of S) and the rest
// o; the pass's flips change w only and keep its popcount k.  So for one k
// and a few words o of popcount nup - k the values x(w, o) form a closed
// set: a tile [C(|S|, k) rows][columns o], staged once in shared memory,
// where every flip is a row index that is the same for all columns and all
// tiles of that k (Sec. 5.3 prefix/postfix view with a window in the place
// of the prefix).
//
// Memory order: the words of the block ascend, so the lowest sites vary
// fastest.  Either S holds the c0 >= 4 lowest sites (rows: consecutive
// window words are consecutive in memory) or it holds none of them
// (columns: consecutive words o are).  Sites 0..3 are therefore taken into a
// window all together or not at all.
#pragma once

#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <map>
#include <vector>

#include "xd_layout.h"

#ifdef __CUDACC__
#define XD_HD __host__ __device__ __forceinline__
#else
#define XD_HD inline
#endif

namespace xd {

constexpr int kWinSites = 12;    // most sites of a window: C(12, 6) = 924 rows
constexpr int kWinLow = 4;       // the sites that are in a window together
constexpr int kWinMaxBonds = 63; // bonds of a pass (6 bits of a list entry, one value left for padding)
constexpr int kWinMaxGroups = 4; // couplings of a pass whose flips are listed coupling by coupling
constexpr int kWinSlots = 1024;  // most row slots of a tile, its zero rows included
// The value types of a product, and the columns of their tiles: 64 bytes of
// values under one window word, a column being one word o (eight values of it in
// the last).
enum WinForm { kWinF64, kWinF32, kWinF32x8, kWinForms };
constexpr int kWinCols[kWinForms] = {8, 16, 2};
constexpr int kWinRows = 16;     // rows of a warp step: two to each lane of four that share a row's columns

struct WinPass {
    std::vector<int> S;          // window sites, ascending
    std::vector<int> bonds;      // the pass's bonds, indices into the distinct pairs
    bool rows = false;           // S holds the lowest sites
    int c0 = 0;                  // how many lowest sites lie inside (rows) or outside S
    std::vector<int> olo, ohi;   // the sites outside S: the lowest c (columns: sites 0..c-1), the others
};

inline uint64_t win_deposit(uint64_t w, const std::vector<int> &sites) {
    uint64_t s = 0;
    for (size_t i = 0; i < sites.size(); ++i) s |= ((w >> i) & 1ull) << sites[i];
    return s;
}

// The distinct site pairs of a bond list and the pair of every bond.
inline std::vector<std::pair<int, int>> win_pairs(const int32_t *bonds, int nb, std::vector<int> *of) {
    std::vector<std::pair<int, int>> out;
    std::map<std::pair<int, int>, int> at;
    of->assign(nb, 0);
    for (int b = 0; b < nb; ++b) {
        const std::pair<int, int> p{std::min(bonds[2 * b], bonds[2 * b + 1]), std::max(bonds[2 * b], bonds[2 * b + 1])};
        auto it = at.find(p);
        if (it == at.end()) {
            it = at.insert({p, (int)out.size()}).first;
            out.push_back(p);
        }
        (*of)[b] = it->second;
    }
    return out;
}

// Mean flips of a row for n bonds.
inline double win_flips(int N, int nup, int n) { return N > 1 ? 2.0 * n * nup * (N - nup) / (N * (N - 1.0)) : 0.0; }

// Share of a tile's columns that are in use when the columns are runs of
// `co` consecutive words of the c lowest sites (win_segments).
inline double win_column_use(int N, int nup, int c, int co) {
    double used = 0, slots = 0;
    for (int m = 0; m <= c; ++m) {
        const double rows = (double)n_choose_k(N - c, nup - m);
        const double cm = (double)n_choose_k(c, m);
        used += rows * cm;
        if (cm >= co) slots += rows * co * (double)(((int64_t)cm + co - 1) / co);
        else slots += rows * co / (cm * 2 <= co ? 2 : 1);
    }
    return slots > 0 ? used / slots : 1.0;
}

// Windows that cover every pair, greedily: each takes the window that covers
// the most uncovered pairs, ties by the fewest sites the remaining pairs
// touch.  Candidates are grown from every site by the site (or the low unit)
// with the most uncovered pairs into the set, and the runs of consecutive
// sites.  Several orders of ties, and of the two criteria, are tried; the cover with the fewest windows
// is kept, then the one whose runs in memory are the longest.  A window with
// room left takes sites that lengthen or keep its runs, so that its tiles
// have rows enough.
inline std::vector<WinPass> choose_windows(int N, int nup, const std::vector<std::pair<int, int>> &pairs) {
    const int W = kWinSites, n = (int)pairs.size();
    const uint64_t low = (1ull << kWinLow) - 1, all = (1ull << N) - 1;
    auto pop = [](uint64_t v) { return __builtin_popcountll(v); };
    auto unit = [&](int v) { return v < kWinLow ? low : 1ull << v; };
    auto runs = [&](uint64_t S, bool *rows) {  // contiguous low sites inside / outside S
        *rows = S & 1;
        const uint64_t t = *rows ? ~S : S;
        return t ? std::min(__builtin_ctzll(t), N) : N;
    };
    using Adj = std::vector<uint64_t>;  // per site: the sites of its uncovered pairs
    Adj full(N, 0);
    for (const auto &p : pairs) {
        full[p.first] |= 1ull << p.second;
        full[p.second] |= 1ull << p.first;
    }
    std::vector<uint64_t> best;
    double best_cost = 0;
    int deg[64], near[64];
    // no window covers more pairs than the best one does at the start
    int most = 1;
    for (int trial = 0, quiet = 0; trial < 96 && quiet < 24; ++trial, ++quiet) {
        uint64_t rng = 0x9E3779B97F4A7C15ull * (uint64_t)(trial + 1);
        auto next = [&]() {
            rng ^= rng << 13;
            rng ^= rng >> 7;
            rng ^= rng << 17;
            return (uint32_t)(rng >> 32);
        };
        Adj a = full;
        std::vector<uint64_t> wins;
        int left = n;
        while (left > 0 && (best.empty() || wins.size() < best.size())) {  // as many windows as the best, or fewer
            uint64_t open = 0;  // sites of uncovered pairs
            int low_pairs = 0, nopen = 0;
            for (int v = 0; v < N; ++v) {
                deg[v] = pop(a[v]);
                open |= (uint64_t)(a[v] != 0) << v;
                nopen += a[v] != 0;
                if (v < kWinLow) low_pairs += pop(a[v] & low);
            }
            int bc = 0, b1 = -(1 << 30), b2 = 0;
            uint32_t bl = 0;
            uint64_t bs = 0;
            // near: per site its uncovered pairs with S, kept as S grows
            auto grow = [&](uint64_t u) {
                for (uint64_t t = u & open; t; t &= t - 1)
                    for (uint64_t q = a[__builtin_ctzll(t)]; q; q &= q - 1) ++near[__builtin_ctzll(q)];
            };
            auto consider = [&](uint64_t S) {
                int cnt = 0, r = nopen;  // uncovered pairs inside S, sites that the others touch
                for (uint64_t t = S & open; t; t &= t - 1) {
                    const int v = __builtin_ctzll(t);
                    cnt += near[v];
                    r -= near[v] == deg[v];
                }
                cnt /= 2;
                if (cnt == 0) return;
                bool rows = false;
                const uint32_t tie = trial == 0 ? (uint32_t)std::min(runs(S, &rows), 8) : next() & 0xffffu;
                const bool sites = trial & 1;  // odd trials: the fewest sites left first
                const int p1 = sites ? -r : cnt, p2 = sites ? cnt : -r;
                if (p1 > b1 || (p1 == b1 && (p2 > b2 || (p2 == b2 && tie > bl)))) {
                    bc = cnt;
                    b1 = p1;
                    b2 = p2;
                    bl = tie;
                    bs = S;
                }
            };
            for (int v0 = 0; v0 < N; ++v0) {
                uint64_t S = unit(v0);
                for (int v = (v0 + 1) % N; pop(S | unit(v)) <= W && v != v0; v = (v + 1) % N) S |= unit(v);
                std::fill(near, near + N, 0);
                grow(S);
                consider(S);
            }
            for (int start = 0; start < N; ++start) {
                if (!a[start]) continue;
                uint64_t S = 0;
                int size = 0;
                std::fill(near, near + N, 0);
                for (uint64_t bu = unit(start); bu;) {
                    S |= bu;
                    size += bu == low ? kWinLow : 1;
                    grow(bu);
                    bu = 0;
                    int bg = 0;
                    auto offer = [&](uint64_t u, int g, int d) {
                        // pairs gained first, then the remaining degree (trial 0) or chance
                        const int score = g * 4096 + (trial == 0 ? d * 16 : (int)(next() & 1023u)) + 1;
                        if (g > 0 && score > bg) {
                            bg = score;
                            bu = u;
                        }
                    };
                    if (!(S & low) && size + kWinLow <= W) {
                        int g = low_pairs, d = 0;
                        for (int v = 0; v < std::min(N, kWinLow); ++v) {
                            g += 2 * near[v];
                            d += deg[v];
                        }
                        offer(low, g, d);
                    }
                    if (size < W)
                        for (uint64_t t = ~S & all & ~low; t; t &= t - 1) {
                            const int v = __builtin_ctzll(t);
                            offer(1ull << v, 2 * near[v], deg[v]);
                        }
                }
                consider(S);
            }
            for (int v = 0; v < N; ++v)
                if ((bs >> v) & 1) a[v] &= ~bs;
            left -= bc;
            wins.push_back(bs);
            if (wins.size() == 1) most = std::max(most, bc);
        }
        if (left > 0) continue;
        double cost = 0;
        for (uint64_t S : wins) {
            bool rows = false;
            const int c0 = runs(S, &rows);
            // short runs move more 32-byte sectors than they use; unused columns are wasted work
            cost += 1.0 + (c0 < 8 ? 0.1 * (8 - c0) : 0.0) + (rows ? 0.0 : 1.0 - win_column_use(N, nup, std::min(c0, 12), 8));
        }
        const size_t before = best.size();
        if (best.empty() || wins.size() < before || cost < best_cost - 1e-9) {
            best = wins;
            best_cost = cost;
        }
        // while fewer windows may do, go on; then a few more for better runs
        if ((int)best.size() > (n + most - 1) / most || best.size() < before) quiet = 0;
        else if (best_cost < (double)best.size() + 0.03) break;  // no window fewer, and little better runs
    }
    std::vector<WinPass> out;
    std::vector<char> cov(n, 0);
    int left = n;
    for (size_t q = 0; left > 0; ++q) {  // a window of more than kWinMaxBonds pairs is done again
        const uint64_t win = best[q % best.size()];
        WinPass p;
        uint64_t S = 0;  // the sites in use (the low unit stays whole)
        for (int t = 0; t < n && (int)p.bonds.size() < kWinMaxBonds; ++t)
            if (!cov[t] && ((win >> pairs[t].first) & (win >> pairs[t].second) & 1ull)) {
                p.bonds.push_back(t);
                cov[t] = 1;
                --left;
                S |= unit(pairs[t].first) | unit(pairs[t].second);
            }
        if (p.bonds.empty()) continue;
        if (S & 1) {
            for (int v = 0; v < N && pop(S) < W; ++v) S |= 1ull << v;
        } else {
            const int c0 = runs(S, &p.rows);
            for (int v = N - 1; v >= std::min(c0, 12) && pop(S) < W; --v) S |= 1ull << v;
        }
        S &= all;
        p.c0 = runs(S, &p.rows);
        std::vector<int> O;
        for (int v = 0; v < N; ++v) ((S >> v) & 1 ? p.S : O).push_back(v);
        int c = std::min({p.c0, 12, (int)O.size()});
        if (p.rows) {
            c = std::min(12, (int)O.size());
        } else {
            for (int t = c - 1; t >= std::min(c, kWinLow); --t)
                if (win_column_use(N, nup, t, 8) > win_column_use(N, nup, c, 8) + 0.02) c = t;
        }
        p.olo.assign(O.begin(), O.begin() + c);
        p.ohi.assign(O.begin() + c, O.end());
        out.push_back(p);
    }
    // the first pass reads no partial sums: the one with the shortest runs goes first
    std::stable_sort(out.begin(), out.end(), [](const WinPass &a, const WinPass &b) { return a.c0 < b.c0; });
    return out;
}

// Estimate of the FP32 product's time per row at half filling, in femtoseconds:
// 4300 a pass (1.4 times that where the lowest sites in the window are few,
// 1.9 times where the columns are runs of the lowest four sites) and 250 a
// flip, fitted to chains, ladders and lattices of 24 to 32 sites.
inline double win_cost32(int N, int nup, const std::vector<WinPass> &passes, int npairs) {
    double c = 250.0 * win_flips(N, nup, npairs);
    for (const WinPass &p : passes) c += 4300.0 * (p.rows ? (p.c0 < 6 ? 1.4 : 1.0) : p.olo.size() <= kWinLow ? 1.9 : 1.0);
    return c;
}

// Words of `sites` by (popcount, value), deposited; off[j] = first of popcount j.
inline void win_words(const std::vector<int> &sites, int jmin, int jmax, std::vector<uint64_t> *words,
                      std::vector<uint32_t> *off) {
    const int n = (int)sites.size();
    off->assign(n + 2, 0);
    for (int j = 0; j <= n; ++j)
        (*off)[j + 1] = (*off)[j] + (j >= jmin && j <= jmax ? (uint32_t)n_choose_k(n, j) : 0u);
    words->assign((*off)[n + 1], 0);
    std::vector<uint32_t> at(off->begin(), off->end() - 1);
    // the words of popcount j ascending: the next word with the same number of ones
    for (int j = std::max(0, jmin); j <= std::min(n, jmax); ++j) {
        uint64_t w = (1ull << j) - 1;
        for (int64_t q = n_choose_k(n, j); q > 0; --q) {
            (*words)[at[j]++] = win_deposit(w, sites);
            if (j == 0) break;
            const uint64_t c = w & (~w + 1), r = w + c;
            w = (((r ^ w) >> 2) / c) | r;
        }
    }
}

// One popcount of a pass's window.
struct WinK {
    int32_t nrows;   // C(|S|, k)
    int32_t nstep;   // groups of kWinRows row slots; the two slots after them are zero rows
    int32_t slot0;   // first entry of this k in the per-slot arrays
    int32_t row0;    // first entry in the per-row array
    int32_t step0;   // first group header
    int32_t list0, nlist;  // flip lists, in 32-bit words
    int32_t whi0, nwhi;    // rows kind: the high parts w >> c0 of this k's words
    int32_t pad;
};

// Tiles of one (k, popcount m of the o_lo word): units of `co` columns, G
// units to a tile.  A unit is chunk q of the C(c, m) words of o_lo under one
// o_hi word, or, where C(c, m) is at most half of co, all of them under two
// consecutive o_hi words.
struct WinSeg {
    int64_t item0;   // first tile
    int64_t units;
    int32_t k, m;
    int32_t hi0, nhi;    // the o_hi words
    int32_t nchunk, per; // chunks to an o_hi word; o_hi words to a unit (1 or 2)
    int32_t cc, cm;      // columns under one o_hi word; C(c, m)
    int32_t G, pad;
};

struct WinTables {
    int ws = 0;
    std::vector<WinK> k;                 // [ws + 1]
    std::vector<uint16_t> slot_word;     // per slot: the window word, 0xffff for none
    std::vector<uint64_t> slot_dep;      // per slot: its word's bits at their sites, ~0 for none
    std::vector<uint64_t> whi;           // rows kind, per k: the high parts w >> c0 of its words, ascending, each with the
                                         // smallest low part, at their sites
    std::vector<uint32_t> rinfo;         // per row, ascending words: slot | place of w >> c0 in whi << 10 | rank of
                                         // the low c0 bits << 18
    std::vector<uint64_t> ohi, olo;      // deposited words by (popcount, value)
    std::vector<uint32_t> ohi_off, olo_off;
    std::vector<uint32_t> list;          // per k, group, four entries: the rows' entries, two words each
    std::vector<uint32_t> step;          // per group of rows: first four of its lists, counts (one byte per coupling)
    int maxslots = 0, maxlist = 0, maxstep = 0;
};


// v / d while v d < 2^20, with inv = win_inv(d): a multiplication and a shift.
XD_HD uint32_t win_inv(uint32_t d) { return ((1u << 20) + d - 1) / d; }
XD_HD uint32_t win_div(uint32_t v, uint32_t inv) { return (v * inv) >> 20; }

// A CTA's tiles are runs of consecutive tiles (n from `tile` on, the first in
// segment seg), so that the lists are loaded once per run, neighbouring tiles
// share their rows' offsets and memory is walked in order.
struct WinRun {
    int64_t tile;
    int32_t n, seg;
};
// A CTA: its runs, its number of tiles and the popcount of the first.
struct WinCta {
    int32_t run0, ntiles, k0, pad;
};

// A tile: its segment (seg: where to start looking, kept from the CTA's tile
// before), its G units, o_hi word uh and chunk ur of the first.  q0, nc0: rank
// of a lone unit's first column and its columns in use (lone: row offsets then
// leave q0 out, so that the tiles of one o_hi word share them); gen: number of
// the row offsets it takes.
struct alignas(16) WinTile {
    int seg, k, m, G;
    int nstep, nslot, nwhi, per;
    int cc, cm, nchunk, hi0;
    int64_t uh;
    int nhi, ur;
    uint32_t inv_chunk, inv_unit;  // inv_unit: rows of a unit (columns kind) or its high parts (rows kind)
    uint32_t inv_step;
    int q0;
    int nc0, gen, fresh, lone;
};

// First column of unit g's o_hi word h (0 or 1): the o_hi word and the rank of
// the o_lo word; the columns that follow under this o_hi word are the next
// ranks, *n of them.  n <= 0 where there is no such word.
XD_HD void win_unit(const WinTile &T, int g, int h, int co, int64_t *hi, int *q, int *n) {
    if (T.nchunk == 1) {
        *hi = T.uh + (T.per == 2 ? 2 * g + h : g);
        *q = 0;
    } else {
        const uint32_t r = (uint32_t)(T.ur + g), dh = win_div(r, T.inv_chunk);
        *hi = T.uh + dh;
        *q = (int)(r - dh * (uint32_t)T.nchunk) * co;
    }
    *n = *hi < T.nhi ? (T.cc < T.cm - *q ? T.cc : T.cm - *q) : 0;
}

// Where a CTA stands in its runs.
struct WinWalk {
    int run, left;
    int64_t tile;
};

// The CTA's next tile.  Before its first: W = {its run0, 0, 0}, T->gen = -1.
// The row offsets are new (fresh) unless the tile before, of the same run and
// segment, was a lone unit under the same o_hi word.
XD_HD void win_next(const WinRun *runs, const WinSeg *segs, int nseg, const WinK *ks, bool rows, int co, WinWalk *W,
                    WinTile *T) {
    int seg0 = T->seg;
    const int64_t uh0 = T->uh;
    if (W->left == 0) {
        W->tile = runs[W->run].tile;
        W->left = runs[W->run].n;
        T->seg = runs[W->run].seg;
        ++W->run;
        seg0 = -1;
    }
    --W->left;
    const int64_t t = W->tile++;
    while (T->seg + 1 < nseg && segs[T->seg + 1].item0 <= t) ++T->seg;
    const WinSeg &s = segs[T->seg];
    const WinK &K = ks[s.k];
    T->k = s.k;
    T->m = s.m;
    T->per = s.per;
    T->cc = s.cc;
    T->cm = s.cm;
    T->nchunk = s.nchunk;
    T->hi0 = s.hi0;
    T->nhi = s.nhi;
    T->nstep = K.nstep;
    T->nslot = kWinRows * K.nstep + 2;
    T->nwhi = K.nwhi;
    const int64_t u0 = (t - s.item0) * s.G, left = s.units - u0;
    T->G = left < s.G ? (int)left : s.G;
    if (s.per == 2) {
        T->uh = 2 * u0;
        T->ur = 0;
    } else if (s.nchunk == 1) {
        T->uh = u0;
        T->ur = 0;
    } else {
        T->uh = (u0 >> 32) ? u0 / s.nchunk : (int64_t)((uint32_t)u0 / (uint32_t)s.nchunk);
        T->ur = (int)(u0 - T->uh * s.nchunk);
    }
    T->inv_chunk = win_inv((uint32_t)s.nchunk);
    T->inv_unit = win_inv((uint32_t)(rows ? K.nwhi : kWinRows * K.nstep));
    T->inv_step = win_inv((uint32_t)K.nstep);
    const int lone0 = T->lone;
    T->lone = !rows && T->G == 1 && s.per == 1;
    int64_t hi;
    win_unit(*T, 0, 0, co, &hi, &T->q0, &T->nc0);
    if (!T->lone) T->q0 = 0;
    T->fresh = !(T->lone && lone0 && seg0 == T->seg && uh0 == T->uh);
    T->gen += T->fresh;
}

// Two-colouring of the window's sites that many bonds cross: the parity of
// the up spins on one colour changes with those bonds' flips and stays with
// the others', which the slots' parities below are taken from.
inline uint32_t win_colour(int ws, const std::vector<uint32_t> &masks) {
    uint32_t best = 0;
    int bn = -1;
    for (int start = 0; start < 2; ++start) {
        uint32_t A = start ? 0x55555555u & ((1u << ws) - 1) : 0;
        for (int sweep = 0; sweep < 32; ++sweep) {
            bool moved = false;
            for (int v = 0; v < ws; ++v) {
                int in = 0, cut = 0;
                for (uint32_t m : masks)
                    if ((m >> v) & 1) {
                        if (__builtin_popcount(A & m) == 1) ++cut;
                        else ++in;
                    }
                if (in > cut) {
                    A ^= 1u << v;
                    moved = true;
                }
            }
            if (!moved) break;
        }
        int n = 0;
        for (uint32_t m : masks) n += __builtin_popcount(A & m) == 1;
        if (n > bn) {
            bn = n;
            best = A;
        }
    }
    return best;
}

// Shared-memory place of a 64-byte row inside its unit: its 16-byte chunk c
// lies at win_row_off ^ (c 16).  Rows kind: the chunks rotate with the slot,
// because neighbouring lanes copy one column of rows in scattered slots.
XD_HD uint32_t win_row_off(bool rows, uint32_t slot) {
    return rows ? slot * 64u | (((slot >> 1) & 3u) << 4) : slot * 64u;
}

// Row slots and flip lists of a pass.  gid[b] (b over the pass's bonds) is
// the bond's coupling group, ng of them; ng = 0: the entries carry the bond.
// Rows whose flips are alike (the same numbers of flips per group) share a
// warp step; a step takes as many rows of either colour parity, alternating,
// so that the row of an even slot and its odd neighbour always read rows of
// opposite parity: the 64-byte rows of a quarter warp then fall into
// different halves of the banks.  Lists are padded inside a step by reads of
// a zero row of the same parity.
struct WinClasses {
    std::vector<uint32_t> masks;  // of the pass's bonds, in window bits
    uint32_t colour = 0;
    std::vector<std::vector<uint32_t>> words;  // per popcount, ascending
};

inline WinClasses win_classes(const WinPass &p, const std::vector<std::pair<int, int>> &pairs) {
    WinClasses c;
    const int ws = (int)p.S.size(), nwb = (int)p.bonds.size();
    c.masks.assign(nwb, 0);
    for (int b = 0; b < nwb; ++b) {
        const auto &pr = pairs[p.bonds[b]];
        for (int i = 0; i < ws; ++i)
            if (p.S[i] == pr.first || p.S[i] == pr.second) c.masks[b] |= 1u << i;
    }
    c.colour = win_colour(ws, c.masks);
    c.words.resize(ws + 1);
    for (uint32_t w = 0; w < (1u << ws); ++w) c.words[__builtin_popcount(w)].push_back(w);
    return c;
}

// The sizes of a pass's tables, which do not depend on the couplings, and the
// high parts of its words.
inline void win_shape(const WinPass &p, const WinClasses &c, WinTables *T) {
    const int ws = (int)p.S.size();
    T->ws = ws;
    T->k.assign(ws + 1, WinK{});
    T->whi.clear();
    T->maxslots = T->maxstep = 0;
    int row0 = 0, slot0 = 0;
    for (int k = 0; k <= ws; ++k) {
        WinK &K = T->k[k];
        int odd = 0;
        for (uint32_t w : c.words[k]) odd += __builtin_popcount(w & c.colour) & 1;
        K.nrows = (int)c.words[k].size();
        K.nstep = (2 * std::max(odd, K.nrows - odd) + kWinRows - 1) / kWinRows;
        K.slot0 = slot0;
        K.row0 = row0;
        slot0 += kWinRows * K.nstep;
        row0 += K.nrows;
        T->maxslots = std::max(T->maxslots, kWinRows * K.nstep + 2);
        T->maxstep = std::max(T->maxstep, K.nstep);
        if (!p.rows) continue;
        K.whi0 = (int)T->whi.size();
        for (size_t i = 0; i < c.words[k].size(); ++i) {
            const uint32_t hi = c.words[k][i] >> p.c0;
            if (i == 0 || hi != c.words[k][i - 1] >> p.c0)
                T->whi.push_back(win_deposit(hi << p.c0 | ((1u << (k - __builtin_popcount(hi))) - 1), p.S));
        }
        K.nwhi = (int)T->whi.size() - K.whi0;
    }
}

inline void win_lists(const WinPass &p, const std::vector<std::pair<int, int>> &pairs, const std::vector<int> &gid,
                      int ng, WinTables *T) {
    const WinClasses cl = win_classes(p, pairs);
    win_shape(p, cl, T);
    const int ws = (int)p.S.size(), nwb = (int)p.bonds.size(), nsub = 2 * std::max(1, ng);
    const std::vector<uint32_t> &masks = cl.masks;
    uint64_t sub[2 * kWinMaxGroups] = {};  // the bonds of a group whose flips change the parity, and keep it
    uint64_t at_site[kWinSites] = {};
    for (int b = 0; b < nwb; ++b) {
        sub[2 * (ng ? gid[b] : 0) + (__builtin_popcount(cl.colour & masks[b]) == 1 ? 0 : 1)] |= 1ull << b;
        for (uint32_t t = masks[b]; t; t &= t - 1) at_site[__builtin_ctz(t)] |= 1ull << b;
    }
    // a word's flipping bonds have one site up: the XOR of the bonds at its up sites
    std::vector<uint64_t> flips(1u << ws, 0), dep(1u << ws, 0);
    for (uint32_t w = 1; w < (1u << ws); ++w) {
        const int v = __builtin_ctz(w);
        flips[w] = flips[w & (w - 1)] ^ at_site[v];
        dep[w] = dep[w & (w - 1)] | 1ull << p.S[v];
    }
    const size_t nslots = T->k[ws].slot0 + kWinRows * T->k[ws].nstep;
    T->slot_word.assign(nslots, 0xffffu);
    T->slot_dep.assign(nslots, ~0ull);
    T->list.clear();
    T->step.clear();
    T->maxlist = 0;
    T->rinfo.assign(1u << ws, 0);
    std::vector<uint16_t> slot_of(1u << ws, 0);
    std::vector<uint64_t> cls[2];  // per parity: the numbers of flips (six bits each), then the word
    constexpr uint64_t kWord = (1ull << kWinSites) - 1;
    static_assert(6 * 2 * kWinMaxGroups + kWinSites <= 64 && kWinMaxBonds < 64, "counts and word in 64 bits");
    for (int k = 0; k <= ws; ++k) {
        WinK &K = T->k[k];
        const std::vector<uint32_t> &words = cl.words[k];
        for (auto &c : cls) c.clear();
        for (uint32_t w : words) {
            uint64_t key = 0;
            for (int s = 0; s < nsub; ++s) key = key << 6 | (uint64_t)__builtin_popcountll(flips[w] & sub[s]);
            cls[__builtin_popcount(w & cl.colour) & 1].push_back(key << kWinSites | w);
        }
        for (auto &c : cls) std::sort(c.begin(), c.end());
        K.step0 = (int)T->step.size() / 2;
        K.list0 = (int)T->list.size();
        for (int c = 0; c < 2; ++c)
            for (size_t i = 0; i < cls[c].size(); ++i) {
                const int slot = 2 * (int)i + c;
                const uint32_t w = (uint32_t)(cls[c][i] & kWord);
                T->slot_word[K.slot0 + slot] = (uint16_t)w;
                T->slot_dep[K.slot0 + slot] = dep[w];
                slot_of[w] = (uint16_t)slot;
            }
        uint32_t pos = 0;  // fours of entries written for this k
        for (int o = 0; o < K.nstep; ++o) {
            const uint16_t *words_at = &T->slot_word[K.slot0 + kWinRows * o];
            int mx[2 * kWinMaxGroups] = {};
            for (int r = 0; r < kWinRows; ++r)
                for (int s = 0; s < nsub && words_at[r] != 0xffffu; ++s)
                    mx[s] = std::max(mx[s], __builtin_popcountll(flips[words_at[r]] & sub[s]));
            T->step.push_back(pos);
            uint32_t counts = 0;
            for (int g = 0; g < nsub / 2; ++g) {
                const int m = mx[2 * g] + mx[2 * g + 1];
                counts |= (uint32_t)m << (8 * g);
                T->list.resize(K.list0 + (size_t)(pos + (m + 3) / 4) * 2 * kWinRows, 0);
                for (int r = 0; r < kWinRows; ++r) {
                    // flips that change the parity first
                    const uint32_t z0 = (uint32_t)(kWinRows * K.nstep) + ((r & 1) ^ 1), z1 = (uint32_t)(kWinRows * K.nstep) + (r & 1);
                    const uint32_t pad0 = ng ? win_row_off(p.rows, z0) : (z0 | (uint32_t)kWinMaxBonds << 10);
                    const uint32_t pad1 = ng ? win_row_off(p.rows, z1) : (z1 | (uint32_t)kWinMaxBonds << 10);
                    uint32_t *at = &T->list[K.list0 + (size_t)pos * 2 * kWinRows + 2 * r];
                    const uint32_t w = words_at[r];
                    int e = 0;
                    for (int keep = 0; keep < 2; ++keep) {
                        uint64_t t = w == 0xffffu ? 0 : flips[w] & sub[2 * g + keep];
                        for (int i = 0; i < mx[2 * g + keep]; ++i, ++e) {
                            uint32_t v = keep ? pad1 : pad0;
                            if (t) {
                                const int b = __builtin_ctzll(t);
                                const uint32_t s = slot_of[w ^ masks[b]];
                                v = ng ? win_row_off(p.rows, s) : (s | (uint32_t)b << 10);
                                t &= t - 1;
                            }
                            at[e / 4 * 2 * kWinRows + ((e >> 1) & 1)] |= v << (16 * (e & 1));
                        }
                    }
                }
                pos += (uint32_t)(m + 3) / 4;
            }
            T->step.push_back(counts);
        }
        K.nlist = (int)T->list.size() - K.list0;
        T->maxlist = std::max(T->maxlist, K.nlist);
        if (p.rows) {
            uint32_t fill[kWinSites + 1] = {}, at = 0;
            const uint32_t lm = (1u << p.c0) - 1;
            for (size_t i = 0; i < words.size(); ++i) {
                if (i > 0 && words[i] >> p.c0 != words[i - 1] >> p.c0) {  // words ascend: ranks restart with the high part
                    ++at;
                    std::fill(fill, fill + kWinSites + 1, 0u);
                }
                const uint32_t rank = fill[__builtin_popcount(words[i] & lm)]++;
                T->rinfo[K.row0 + i] = (uint32_t)slot_of[words[i]] | at << 10 | rank << 18;
            }
        }
    }
}

// The words outside the window.
inline void win_outer(const WinPass &p, int nup, WinTables *T) {
    const int ws = (int)p.S.size(), c = (int)p.olo.size();
    win_words(p.ohi, nup - ws - c, nup, &T->ohi, &T->ohi_off);
    win_words(p.olo, 0, c, &T->olo, &T->olo_off);
}

// Tiles of a pass with co columns, taken k by k; at most `ctas` tiles' worth
// of units are put into one tile, so that a small block spreads over the
// chip.  nbase: most row offsets that a tile keeps.
constexpr int kWinBase = 2048;

inline std::vector<WinSeg> win_segments(const WinPass &p, const WinTables &T, int nup, int co, int ctas,
                                        int64_t *nitems, int *nbase) {
    const int ws = (int)p.S.size(), c = (int)p.olo.size(), nh = (int)p.ohi.size();
    std::vector<WinSeg> out;
    int64_t item = 0;
    *nbase = 0;
    for (int k = 0; k <= ws; ++k) {
        for (int m = 0; m <= c; ++m) {
            const int j = nup - k - m;
            if (j < 0 || j > nh) continue;
            WinSeg s{};
            s.item0 = item;
            s.k = k;
            s.m = m;
            s.hi0 = (int)T.ohi_off[j];
            s.nhi = (int)n_choose_k(nh, j);
            s.cm = (int)n_choose_k(c, m);
            s.cc = std::min(s.cm, co);
            const int rows = kWinRows * T.k[k].nstep;
            // two o_hi words side by side cost a second row offset per row: where few rows or short runs make it worth it
            s.per = 2 * s.cm <= co && (p.rows || c <= kWinLow || 2 * rows <= T.maxslots) ? 2 : 1;
            s.nchunk = (s.cm + co - 1) / co;
            s.units = s.per == 2 ? (s.nhi + 1) / 2 : (int64_t)s.nhi * s.nchunk;
            if (s.units == 0) continue;
            const int entries = p.rows ? T.k[k].nwhi * co : rows * s.per;
            s.G = (int)std::max<int64_t>(1, std::min({(int64_t)(T.maxslots / (rows + 2)), (int64_t)(kWinBase / entries),
                                                      (int64_t)64, (s.units + ctas - 1) / ctas}));
            *nbase = std::max(*nbase, s.G * entries);
            item += (s.units + s.G - 1) / s.G;
            out.push_back(s);
        }
    }
    *nitems = item;
    return out;
}

// 64-bit row offsets
inline bool win_wide(int64_t dim) { return dim >= (int64_t)0xffffffffll; }

// The shared memory of a CTA: two tiles, the flip lists and step headers of one
// popcount, the coefficients, (rows kind) the rows, and three sets of row
// offsets, or two where three do not fit.  T: maxslots, maxlist, maxstep; nbase:
// of win_segments; wide: 64-bit row offsets.
constexpr uint32_t kWinSmem = 225 * 1024;  // of the 227 KB a CTA can have; the kernel keeps 1.3 KB of its own

struct WinSmem {
    uint32_t tile1, list, step, coef, rinfo, base, base_bytes, total;
    int base_sets;
    bool fits() const { return total <= kWinSmem; }
};

inline WinSmem win_smem(bool rows, int maxslots, int maxlist, int maxstep, int ncoef, int nbase, bool wide) {
    WinSmem s{};
    uint32_t o = (uint32_t)maxslots * 128;
    auto take = [&](size_t bytes) {
        const uint32_t at = o;
        o += (uint32_t)((bytes + 15) / 16 * 16);
        return at;
    };
    s.tile1 = (uint32_t)maxslots * 64;
    s.list = take((size_t)maxlist * 4);
    s.step = take((size_t)maxstep * 8);
    s.coef = take((size_t)ncoef * 8);
    s.rinfo = take(rows ? kWinSlots * 4 : 0);
    s.base_bytes = (uint32_t)(((size_t)nbase * (wide ? 8 : 4) + 15) / 16 * 16);
    s.base_sets = o + 3 * s.base_bytes <= kWinSmem ? 3 : 2;
    s.base = take((size_t)s.base_sets * s.base_bytes);
    s.total = o;
    return s;
}

// The tiles' division among at most `ctas` CTAs.  Many tiles (kWinMany to a
// CTA): a run of every popcount k, of equal length up to one, the longer ones
// dealt on from k to k; all CTAs then work on tiles of one cost at a time.
// Few: one run, by an estimate of the cost of a tile in clocks (6000 and, for
// every row, 3.5 and 0.6 for each of its flips), because every new k costs the
// loading of its lists, about 12000 clocks.
constexpr int kWinMany = 64;

inline void win_divide(const WinPass &p, const WinTables &T, const std::vector<WinSeg> &segs, int64_t nitems, int ctas,
                       std::vector<WinCta> *cta, std::vector<WinRun> *runs) {
    const int n = (int)std::min<int64_t>(ctas, nitems), ws = (int)p.S.size();
    auto tiles = [&](size_t q) { return (segs[q].units + segs[q].G - 1) / segs[q].G; };
    auto seg_of = [&](int64_t t) {
        size_t q = 0;
        while (q + 1 < segs.size() && segs[q + 1].item0 <= t) ++q;
        return (int32_t)q;
    };
    cta->assign(n + 1, WinCta{0, 0, 0, 0});
    runs->clear();
    std::vector<int64_t> first(n + 1, nitems);
    if (nitems < (int64_t)kWinMany * ctas) {
        std::vector<double> cost(segs.size());
        double all = 0, done = 0;
        for (size_t q = 0; q < segs.size(); ++q) {
            const int k = segs[q].k;
            const double flips = ws > 1 ? 2.0 * p.bonds.size() * k * (ws - k) / (ws * (ws - 1.0)) : 0.0;
            cost[q] = 6000.0 + segs[q].G * kWinRows * T.k[k].nstep * (3.5 + 0.6 * flips);
            all += cost[q] * (double)tiles(q);
        }
        int c = 0;
        for (size_t q = 0; q < segs.size(); ++q) {
            for (; c < n; ++c) {  // it begins at the first tile at or past its share of the cost
                const int64_t t = std::max<int64_t>(0, (int64_t)std::ceil((all * c / n - done) / cost[q] - 1e-9));
                if (t >= tiles(q)) break;
                first[c] = segs[q].item0 + t;
            }
            done += cost[q] * (double)tiles(q);
        }
    }
    std::vector<int64_t> at(ws + 2, nitems);  // first tile of each k
    for (size_t q = segs.size(); q-- > 0;) at[segs[q].k] = segs[q].item0;
    for (int k = ws; k >= 0; --k)
        if (at[k] > at[k + 1]) at[k] = at[k + 1];
    for (int c = 0; c < n; ++c) {
        (*cta)[c].run0 = (int32_t)runs->size();
        auto add = [&](int64_t t, int64_t end) {
            if (t >= end) return;
            runs->push_back(WinRun{t, (int32_t)(end - t), seg_of(t)});
            if ((*cta)[c].ntiles == 0) (*cta)[c].k0 = segs[runs->back().seg].k;
            (*cta)[c].ntiles += (int32_t)(end - t);
        };
        if (nitems < (int64_t)kWinMany * ctas) {
            add(first[c], first[c + 1]);
            continue;
        }
        for (int k = 0; k <= ws; ++k) {
            const int64_t len = at[k + 1] - at[k], each = len / n, rem = len % n, v = ((c - at[k]) % n + n) % n;
            const int64_t t = at[k] + v * each + std::min(v, rem);
            add(t, t + each + (v < rem ? 1 : 0));
        }
    }
    (*cta)[n].run0 = (int32_t)runs->size();
}

// Flip lists of a pass with bonds in ng coupling groups (gid): coupling by
// coupling, or with the bond in each entry (ng = 0).  Every coupling pads its
// part of a step's lists, so that with several of them on a dense graph the
// lists coupling by coupling may not fit in shared memory; the pass then takes
// the entries that carry the bond where these leave room for more value types
// (lists of 63 bonds and four couplings: 96 KB and 72 KB).  Returns the ng
// taken; fit: whether products of each value type fit (64-bit row offsets: none
// on eight vectors).
inline int win_fitting_lists(const WinPass &p, const std::vector<std::pair<int, int>> &pairs, const int *nbase, bool wide,
                             const std::vector<int> &gid, int ng, WinTables *T, bool *fit) {
    auto room = [&](const WinTables &t, int groups, bool *f) {
        int n = 0;
        for (int q = 0; q < kWinForms; ++q) {
            f[q] = !(wide && q == kWinF32x8) &&
                   win_smem(p.rows, t.maxslots, t.maxlist, t.maxstep, groups ? groups : kWinMaxBonds + 1, nbase[q], wide).fits();
            n += f[q];
        }
        return n;
    };
    win_lists(p, pairs, gid, ng, T);
    const int n = room(*T, ng, fit);
    if (ng == 0 || n == (wide ? kWinForms - 1 : (int)kWinForms)) return ng;
    WinTables B;
    bool fb[kWinForms];
    win_lists(p, pairs, std::vector<int>(p.bonds.size(), 0), 0, &B);
    if (room(B, 0, fb) <= n) return ng;
    *T = std::move(B);
    std::copy(fb, fb + kWinForms, fit);
    return 0;
}

// A pass with what does not depend on the couplings: its shape, the words
// outside its window and, for every value type, its tiles and their division.
struct WinPlan {
    WinPass p;
    WinTables T;
    std::vector<WinSeg> segs[kWinForms];
    std::vector<WinCta> ctas[kWinForms];
    std::vector<WinRun> runs[kWinForms];
    int nbase[kWinForms] = {};
};

// The passes of a block on a chip of `sms` CTAs.  A pass whose bond-carrying
// lists would not fit is done in two, each with half of its bonds; FP32 beside
// 64-bit row offsets (twice the room, and twice the columns of FP64) may be
// left without.
inline std::vector<WinPlan> win_plan(int N, int nup, const std::vector<std::pair<int, int>> &pairs, int sms) {
    const bool wide = win_wide(n_choose_k(N, nup));
    std::vector<WinPlan> out;
    std::vector<WinPass> todo = choose_windows(N, nup, pairs);
    std::reverse(todo.begin(), todo.end());
    while (!todo.empty()) {
        WinPlan d;
        d.p = todo.back();
        todo.pop_back();
        const WinPass &p = d.p;
        win_shape(p, win_classes(p, pairs), &d.T);
        win_outer(p, nup, &d.T);
        for (int q = 0; q < kWinForms; ++q) {
            int64_t nitems = 0;
            d.segs[q] = win_segments(p, d.T, nup, kWinCols[q], sms, &nitems, &d.nbase[q]);
            win_divide(p, d.T, d.segs[q], nitems, sms, &d.ctas[q], &d.runs[q]);
        }
        // a list holds at most every bond of the pass: most passes fit at that size
        const int nwb = (int)p.bonds.size(), most = d.T.maxstep * 2 * kWinRows * ((nwb + 3) / 4);
        bool fit[kWinForms], all = true;
        for (int q = 0; q < kWinForms; ++q)
            all = all && win_smem(p.rows, d.T.maxslots, most, d.T.maxstep, kWinMaxBonds + 1, d.nbase[q], wide).fits();
        if (!all && nwb > 1) {
            WinTables T;
            win_fitting_lists(p, pairs, d.nbase, wide, std::vector<int>(nwb, 0), 0, &T, fit);
            if (wide ? !fit[kWinF64] : !(fit[kWinF64] && fit[kWinF32] && fit[kWinF32x8])) {
                WinPass a = p, b = p;
                a.bonds.resize(nwb / 2);
                b.bonds.erase(b.bonds.begin(), b.bonds.begin() + nwb / 2);
                todo.push_back(b);
                todo.push_back(a);
                continue;
            }
        }
        out.push_back(std::move(d));
    }
    return out;
}

}  // namespace xd
