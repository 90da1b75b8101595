// The window product's tables (csrc/xd_window.h) read the way its kernel
// reads them, on the host: every tile's row offsets, staged values, flip
// lists and sums, with every index checked against what it indexes.
#include <stdio.h>

#include "xd_window.h"

using namespace xd;

namespace {

struct Shape {
    int value_bytes, co, nv;
};

// One pass of one value type over all tiles: y += pass(x).  Rows of x hold nv
// values.  Returns 0, or the number of the check that failed.
int run_pass(const WinPass &p, const WinTables &T, const std::vector<double> &coef, int ng, const U1Layout &lay, int nup,
             Shape sh, int ctas_wanted, const double *x, double *y, const std::vector<double> &diag) {
    const int CW = 64 / sh.value_bytes, co = sh.co;
    int64_t nitems = 0;
    std::vector<WinCta> ctas;
    std::vector<WinRun> runs;
    int nbase = 0;
    const std::vector<WinSeg> segs = win_segments(p, T, nup, co, ctas_wanted, &nitems, &nbase);
    win_divide(p, T, segs, nitems, ctas_wanted, &ctas, &runs);
    if (T.maxslots > kWinSlots) return 1;
    std::vector<char> seen((size_t)lay.dim * sh.nv, 0);
    std::vector<double> tile((size_t)T.maxslots * CW);
    // place of a value in the tile: the unit's bytes, then the row's offset (staging: from the slot; flips: from
    // the list entry) with the column's chunk and place in it
    auto at = [&](int unit_bytes, uint32_t row_off, int j) {
        const bool wide = sh.value_bytes == 4 && sh.nv == 8;  // eight FP32 vectors: four neighbours to a chunk
        const uint32_t chunk = (uint32_t)(wide ? j >> 2 : j & 3), in = (uint32_t)((wide ? j & 3 : j >> 2) * sh.value_bytes);
        const uint32_t o = row_off ^ chunk << 4 ^ in;
        return (int64_t)((unit_bytes + o) / sh.value_bytes);
    };
    if (win_div(1023, win_inv(8)) != 127 || win_div(2047, win_inv(255)) != 8) return 19;
    for (size_t cta = 0; cta + 1 < ctas.size(); ++cta) {
    WinTile T1;
    T1.seg = 0;
    T1.gen = -1;
    T1.lone = 0;
    T1.uh = 0;
    WinWalk walk{ctas[cta].run0, 0, 0};
    uint64_t owner = 0;  // the o_hi word of the row offsets in use
    for (int i = 0; i < ctas[cta].ntiles; ++i) {
        win_next(runs.data(), segs.data(), (int)segs.size(), T.k.data(), p.rows, co, &walk, &T1);
        const int64_t t = walk.tile - 1;
        if (i == 0 && T1.k != ctas[cta].k0) return 24;
        if (walk.run > ctas[cta + 1].run0 || t < segs[T1.seg].item0 || t >= nitems) return 20;
        if (T1.seg + 1 < (int)segs.size() && t >= segs[T1.seg + 1].item0) return 21;
        {
            int64_t hi;
            int q, n;
            win_unit(T1, 0, 0, co, &hi, &q, &n);
            const uint64_t o = T.ohi[T1.hi0 + hi];
            if (T1.fresh) owner = o ^ ((uint64_t)T1.k << 58);
            else if (owner != (o ^ ((uint64_t)T1.k << 58)) || T1.G != 1 || T1.q0 != q) return 22;  // shared row offsets: the same o_hi word
            if (T1.nc0 != n) return 23;
        }
        const WinK &K = T.k[T1.k];
        const int nslot = T1.nslot, G = T1.G;
        if (G * nslot > T.maxslots || G > 64 || G * K.nstep > kWinSlots / kWinRows) return 3;
        {
            std::fill(tile.begin(), tile.end(), 0.0);
            std::vector<std::vector<int64_t>> idx(G * kWinRows * K.nstep, std::vector<int64_t>(CW, -1));
            for (int g = 0; g < G; ++g) {
                for (int j = 0; j < CW; ++j) {
                    const int jo = j / sh.nv, v = j % sh.nv;
                    const int h = T1.per == 2 && jo >= T1.cc ? 1 : 0, lr = jo - h * T1.cc;
                    int64_t hi;
                    int q0, nc;
                    win_unit(T1, g, h, co, &hi, &q0, &nc);
                    if (lr >= T1.cc || lr >= nc) continue;
                    const int q = q0 + lr;
                    const uint64_t o = T.ohi[T1.hi0 + hi];
                    if (__builtin_popcountll(o) + T1.k + T1.m != nup) return 2;
                    for (int r = 0; r < K.nrows; ++r) {
                        int slot;
                        int64_t row;
                        if (p.rows) {
                            const uint32_t e = T.rinfo[K.row0 + r];
                            slot = e & 1023u;
                            const int wi = (e >> 10) & 255u;
                            if (wi >= K.nwhi || G * K.nwhi * co > nbase) return 4;
                            if ((int)win_div((uint32_t)(g * K.nwhi + wi), T1.inv_unit) != g) return 17;
                            const uint64_t w = T.whi[K.whi0 + wi] | o | T.olo[T.olo_off[T1.m] + q];
                            row = u1_index((int)lay.L + lay.P, nup, lay.L, lay.hi_off, lay.lo_rank, w);
                            if (row < 0) return 5;
                            row += e >> 18;
                        } else {
                            // rows in slot order
                            if (kWinRows * K.nstep * T1.per * G > nbase) return 6;
                            slot = -1;
                            int c = 0;
                            for (int z = 0; z < kWinRows * K.nstep; ++z)
                                if (T.slot_word[K.slot0 + z] != 0xffffu && c++ == r) slot = z;
                            if (slot < 0) return 7;
                            if ((int)win_div((uint32_t)(g * kWinRows * K.nstep + slot), T1.inv_unit) != g) return 18;
                            const uint64_t w = T.slot_dep[K.slot0 + slot] | o | ((1ull << T1.m) - 1);
                            row = u1_index((int)lay.L + lay.P, nup, lay.L, lay.hi_off, lay.lo_rank, w);
                            if (row < 0) return 8;
                            // as the kernel: the row offset of the unit, then the tile's first rank and the column
                            row += (T1.lone ? 0 : q0) + T1.q0 + lr;
                            if (T1.lone && nc != T1.nc0) return 25;
                        }
                        if (slot >= kWinRows * K.nstep || row < 0 || row >= lay.dim) return 9;
                        const int64_t i = row * sh.nv + v;
                        if (seen[i]) return 10;
                        seen[i] = 1;
                        tile[at(g * nslot * 64, win_row_off(p.rows, (uint32_t)slot), j)] = x[i];
                        idx[g * kWinRows * K.nstep + slot][j] = i;
                    }
                }
            }
            for (int g = 0; g < G; ++g)
                for (int o = 0; o < K.nstep; ++o) {
                    uint32_t pos = T.step[2 * (K.step0 + o)];
                    const uint32_t counts = T.step[2 * (K.step0 + o) + 1];
                    for (int r = 0; r < kWinRows; ++r) {
                        const int slot = kWinRows * o + r;
                        for (int j = 0; j < CW; ++j) {
                            if (idx[g * kWinRows * K.nstep + slot][j] < 0) continue;
                            double a = 0;
                            uint32_t ps = pos;
                            for (int q = 0; q < std::max(1, ng); ++q) {
                                const int n = ng ? (int)((counts >> (8 * q)) & 255u) : (int)counts;
                                for (int e = 0; e < n; ++e) {
                                    const size_t li = (size_t)(ps + e / 4) * 2 * kWinRows + 2 * r + ((e >> 1) & 1);
                                    if ((int)li >= K.nlist) return 11;
                                    const uint32_t v = (T.list[K.list0 + li] >> (16 * (e & 1))) & 0xffffu;
                                    const uint32_t ts = ng ? v >> 6 : v & 1023u;
                                    if ((int)ts >= nslot) return 12;
                                    if (ng && v != win_row_off(p.rows, ts)) return 13;
                                    if (!ng && (int)(v >> 10) >= (int)coef.size()) return 14;
                                    // rows of a pair read rows of opposite parity
                                    const uint32_t o2 = T.list[K.list0 + (li ^ 2)] >> (16 * (e & 1));
                                    if (((ng ? (o2 & 0xffffu) >> 6 : o2 & 1023u) & 1) == (ts & 1)) return 15;
                                    a += coef[ng ? q : (int)(v >> 10)] *
                                         tile[at(g * nslot * 64, ng ? v : win_row_off(p.rows, ts), j)];
                                }
                                ps += (uint32_t)(n + 3) / 4;
                            }
                            const int64_t i = idx[g * kWinRows * K.nstep + slot][j];
                            y[i] += a + diag[T.slot_word[K.slot0 + slot]] * x[i];
                        }
                    }
                }
        }
    }
    }
    for (char c : seen)
        if (!c) return 16;
    return 0;
}

}  // namespace

extern "C" {

// Windows of a graph: returns their number; out[q][13]: rows kind, then the sites (-1 past the end).
int window_sites(int N, int nup, const int32_t *bonds, int nb, int32_t *out, int cap) {
    std::vector<int> of;
    const auto pairs = win_pairs(bonds, nb, &of);
    const auto ps = choose_windows(N, nup, pairs);
    for (int q = 0; q < (int)ps.size() && q < cap; ++q)
        for (int i = 0; i < 13; ++i)
            out[13 * q + i] = i == 0 ? (int)ps[q].rows : i - 1 < (int)ps[q].S.size() ? ps[q].S[i - 1] : -1;
    return (int)ps.size();
}

// y = H x through the tables; value_bytes 8 or 4, nv values per row.  force_bond: lists that carry the bond.
int window_product(int N, int nup, const int32_t *bonds, int nb, const double *J, int value_bytes, int nv, int force_bond,
                   int ctas, const double *x, double *y) {
    U1Layout lay;
    if (!u1_layout(N, nup, &lay)) return 100;
    std::vector<int> of;
    const auto pairs = win_pairs(bonds, nb, &of);
    std::vector<double> Jp(pairs.size(), 0.0);
    for (int b = 0; b < nb; ++b) Jp[of[b]] += J[b];
    std::vector<int> covered(pairs.size(), 0);
    for (int64_t i = 0; i < lay.dim * nv; ++i) y[i] = 0.0;
    for (const WinPass &p : choose_windows(N, nup, pairs)) {
        std::vector<double> vals;
        std::vector<int> gid;
        for (int b : p.bonds) {
            ++covered[b];
            size_t g = std::find(vals.begin(), vals.end(), Jp[b]) - vals.begin();
            if (g == vals.size()) vals.push_back(Jp[b]);
            gid.push_back((int)g);
        }
        if ((int)p.bonds.size() > kWinMaxBonds) return 101;
        const int ng = force_bond || (int)vals.size() > kWinMaxGroups ? 0 : (int)vals.size();
        if (!ng) gid.assign(gid.size(), 0);
        WinTables T;
        win_lists(p, pairs, gid, ng, &T);
        win_outer(p, nup, &T);
        std::vector<double> coef(ng ? ng : kWinMaxBonds + 1, 0.0), diag(1u << p.S.size(), 0.0);
        for (size_t t = 0; t < p.bonds.size(); ++t) {
            const auto &pr = pairs[p.bonds[t]];
            coef[ng ? gid[t] : (int)t] = 0.5 * Jp[p.bonds[t]];
            for (uint32_t w = 0; w < diag.size(); ++w) {
                const uint64_t s = win_deposit(w, p.S);
                diag[w] += (((s >> pr.first) ^ (s >> pr.second)) & 1) ? -0.25 * Jp[p.bonds[t]] : 0.25 * Jp[p.bonds[t]];
            }
        }
        const int rc = run_pass(p, T, coef, ng, lay, nup, Shape{value_bytes, 64 / value_bytes / nv, nv}, ctas, x, y, diag);
        if (rc) return rc;
    }
    for (int c : covered)
        if (c != 1) return 102;
    return 0;
}
}
