// xd_u1_win.cu -- y = H x on large U(1) blocks (large_block) in passes over
// windows of sites.
//
// H = sum of passes, each the bonds inside a window S of at most 12 sites
// (choose_windows, xd_window.h; Sec. 5.3 prefix/postfix view with a window in
// the place of the prefix; Eq. 1, pull form, rows written once per pass, no
// atomics).  The pass's flips change only the bits of S and keep their
// popcount, so the rows that share the other bits form a closed set: a tile
// [C(|S|, k) window words][64 bytes of columns, the words outside S] is
// staged once in shared memory and every flip is one 16-byte shared-memory
// read whose row offset comes from a list that is the same for every tile of
// that k.  Each pass adds its bonds' flips and its share of the diagonal,
//     p(w, o) = sum over flipping b of (J_b / 2) x(w ^ m_b, o) + D_S(w) x(w, o),
//     D_S(w) = sum over the window's bonds of +-J_b / 4,
// to the partial sums kept in y's memory.
//
// What bounds it: the load/store unit of the SM -- one 16-byte read per two
// (FP32: four) matrix elements and lane, and the reads and writes of x and of
// the partial sums, whose 64-byte runs cost a tag lookup each.  Hence the
// layout: four lanes read one 64-byte row; the rows of a quarter warp have
// opposite slot parity (win_lists), so that the reads have no bank conflicts
// (16-byte chunks of random rows otherwise cost 1.8 wavefronts); rows with
// equally long lists share a warp step, so that no lane waits; eight lanes
// share a row when it goes to or comes from memory.  One CTA of 768 threads
// per SM with two tiles in shared memory: 17 warps flip one tile while six
// copy the next and one works out the tile after that (two CTAs of 512
// threads that did everything in turn took 44 ms for the 4x8 lattice in FP64).
// Measured (us; before: prefix blocks, xd_u1_passes.cu and xd_u1_spmm.cu):
//                          FP64            FP64 double-float   FP32
//   4x8 lattice, J1-J2     59500 -> 32000  70200 -> 47700      31800 -> 18100
//   32-site chain          31800 -> 18200  34800 -> 20200      10900 ->  9900
//   28-site ladder          3320 ->  1820   3890 ->  2090       1600 ->  1270
//   24-site lattice 4x6      256 ->   199    294 ->   282        146 ->   138
// At the 4x8 lattice a pass moves 14.4 GB if every value crosses once (2.2 ms at
// the measured copy rate), 17.9 on average by the counters of the 4x7 lattice, and
// takes 5.5 to 9 ms with the load/store unit 58 to 65% busy.
//
// Arithmetic: FP64 input and output (the paper's precision) without FP64
// arithmetic per element (GB300's FP64 pipe is a small fraction of its FP32
// and integer rates), in one of two arithmetics chosen per product on the
// device:
//     fixed point, for couplings that are small integer multiples k_b q of
//     one quantum q (e.g. J1 = 1, J2 = 1/2, any uniform model): in units of
//     q/4 a row is y_r = (q/4) (D(s_r) x_r + sum over flipped b of 2 k_b x_c),
//     D(s) = sum_b k_b eps_b(s) an integer; x is scaled by 2^S and rounded to
//     64-bit integers X (|X| < 2^B, no row sum can overflow) and every sum
//     is exact; each row is converted to FP64 once;
//     double-float, for any couplings: x is scaled by 2^(1023 - E) (E its
//     largest biased exponent) and split into FP32 pairs (hi, lo), hi the
//     top 24 significant bits (exact), lo the next bits rounded to FP32; each
//     coefficient c is a pair (C, gamma); per element c x is p + e exactly
//     (p = fl32(C hi), e = fma(C, hi, -p)) plus the small terms C lo + gamma
//     hi, p enters the accumulator by TwoSum (Knuth) and every rounding error
//     joins the second word; the row's result 2^(E - 1023) (s + c) costs one
//     FP64 addition: a relative error near 2^-45 of the sum of the
//     magnitudes of the row's terms.
//     A statistics pass (largest exponent and a lower bound of |x|) lets the
//     device take double-float whenever rounding x to the fixed-point grid
//     could cost more than 2^-44 |x| (vectors dominated by a few entries).

#include <string.h>

#include <algorithm>
#include <vector>

#include "xd_internal.cuh"
#include "xd_window.h"
#include "xd_x64.cuh"

namespace xd {

namespace {

// ------------------------------------------------------------- arithmetics
// V: staged values; Acc: partial sums (as large as V); C: flip coefficient;
// D: diagonal of a window word; Y: result.  Lists coupling by coupling: list adds
// a value of a coupling's part, mul_add that part's sum with its coefficient; in
// FP32 list multiplies (an FMA costs what an addition does), because a sum of x
// alone can overflow where no J x and no sum of them does.
struct PolDF {
    static constexpr int kArith = 0;
    using V = float2;     // scaled x as (hi, lo)
    using C = float2;     // J/2 as (C, gamma)
    using D = float2;
    using Y = double;
    struct __align__(8) Acc {
        float s, c;
    };
    struct Out {
        int E;
    };
    __device__ static void zero(Acc &a) { a.s = a.c = 0.f; }
    __device__ static void add(Acc &a, V v) {
        const float2 r = df_add(make_float2(a.s, a.c), v);
        a.s = r.x;
        a.c = r.y;
    }
    __device__ static void list(Acc &a, C, V v) { add(a, v); }
    __device__ static void list(Acc &a, C, V v, V w) {
        add(a, v);
        add(a, w);
    }
    __device__ static void mul_add(Acc &a, C c, Acc s) { df_fma(a.s, a.c, c, make_float2(s.s, s.c)); }
    __device__ static void fma(Acc &a, C c, V v) { df_fma(a.s, a.c, c, v); }
    __device__ static void diag(Acc &a, D d, V v) { df_fma(a.s, a.c, d, v); }
    __device__ static void merge(Acc &a, Acc b) { add(a, make_float2(b.s, b.c)); }
    template <class P> __device__ static Out out_setup(const P &, int E) { return Out{E}; }
    __device__ static Y result(Acc a, const Out &o) { return df_result(a.s, a.c, o.E); }
};

struct PolFX {
    static constexpr int kArith = 1;
    using V = long long;  // round(2^S x)
    using C = int;        // 2 k_b, in units of q/4
    using D = int;        // sum_b k_b eps_b(w), in units of q/4
    using Y = double;
    struct Acc {
        long long a;
    };
    struct Out {
        double f;         // (q/4) 2^-S
        bool nan;
    };
    __device__ static void zero(Acc &a) { a.a = 0; }
    __device__ static void list(Acc &a, C, V v) { a.a += v; }
    __device__ static void list(Acc &a, C, V v, V w) { a.a = a.a + v + w; }  // three-input adds
    __device__ static void mul_add(Acc &a, C c, Acc s) { a.a += (long long)c * s.a; }
    __device__ static void fma(Acc &a, C c, V v) { a.a += (long long)c * v; }
    __device__ static void diag(Acc &a, D d, V v) { a.a += (long long)d * v; }
    __device__ static void merge(Acc &a, Acc b) { a.a += b.a; }
    template <class P> __device__ static Out out_setup(const P &p, int E) {
        // S = B - E + 1022: the scaled largest entry is below 2^B
        return Out{pow2d(E - 1022 - p.B, p.qs), E == 2047};
    }
    __device__ static Y result(Acc a, const Out &o) {
        return o.nan ? __longlong_as_double(0x7ff8000000000000ll) : (double)a.a * o.f;
    }
};

struct PolF32 {
    static constexpr int kArith = 2;
    using V = float;
    using C = float;
    using D = float;
    using Y = float;
    struct Acc {
        float a;
    };
    struct Out {};
    __device__ static void zero(Acc &a) { a.a = 0.f; }
    __device__ static void list(Acc &a, C c, V v) { a.a = fmaf(c, v, a.a); }
    __device__ static void list(Acc &a, C c, V v, V w) { a.a = fmaf(c, w, fmaf(c, v, a.a)); }
    __device__ static void mul_add(Acc &a, C, Acc s) { a.a += s.a; }
    __device__ static void fma(Acc &a, C c, V v) { a.a = fmaf(c, v, a.a); }
    __device__ static void diag(Acc &a, D d, V v) { a.a = fmaf(d, v, a.a); }
    __device__ static void merge(Acc &a, Acc b) { a.a += b.a; }
    template <class P> __device__ static Out out_setup(const P &, int) { return Out{}; }
    __device__ static Y result(Acc a, const Out &) { return a.a; }
};

// ------------------------------------------------------------------ kernel
constexpr int kT = 768;     // threads per CTA: kCW warps that flip, one that plans, the others copy
constexpr int kCW = 17;
constexpr int kPT = kT - 32 * kCW - 32;                        // copying threads
constexpr int kMeet = 32 * kCW + kPT;                           // threads that meet over a tile's buffer
constexpr int kSteps = (kWinSlots / kWinRows + kCW - 1) / kCW;  // steps per flipping warp and tile

struct WinParams {
    const int64_t *hi_off;      // the block's two-table index: index(s) = hi_off[s >> L] + lo_rank[s & lomask]
    const uint32_t *lo_rank;
    int L;
    uint32_t lomask;
    const WinK *ks;             // [ws + 1]
    const WinSeg *segs;
    int nseg, c0, co;           // co: columns o of a tile (64 bytes / value size / nv)
    int cos;                    // log2 of co
    const WinCta *ctas;
    const WinRun *runs;
    const uint64_t *slot_dep, *whi, *ohi, *olo;
    const uint32_t *rinfo, *list;
    const uint2 *step;
    const uint32_t *olo_off;
    const void *coef[3];        // [max(ng, bonds + 1)] by coupling group, or by bond (ng = 0), for each arithmetic
    int ncoef, ng;
    const void *diag[3];        // per slot
    int first, last;
    uint32_t sm_tile1, sm_list, sm_step, sm_coef, sm_rinfo, sm_base, base_bytes;
    int nbase_bufs;             // 3, or 2 where three do not fit
    double qs;                  // q/4 (fixed point)
    int B;                      // |X| < 2^B (fixed point)
    const int *state;           // [E, mode]
};

// Row offsets of a tile's parts, ~0 where there is none: columns kind, per
// unit, slot and o_hi word, the first of its consecutive rows (a lone unit's
// without its q0); rows kind, per
// unit, high part of the window word and column, the first of its rows.
// ncol: columns in use of every unit (one o_hi word to a unit).  Four entries
// of a thread at a time, so that their table reads are in flight together.
template <bool ROWS, typename I>
__device__ __forceinline__ void tile_base(const WinParams &p, const WinTile &T, I *base, uint8_t *ncol, int ptid) {
    constexpr int U = 4;
    const int n = ROWS ? T.nwhi : kWinRows * T.nstep, per = T.per, G = T.G, cc = T.cc;
    const int tot = ROWS ? (G * n) << p.cos : G * n * per;
    const uint32_t inv = T.inv_unit;
    const uint64_t *parts = ROWS ? p.whi + __ldg(&p.ks[T.k].whi0) : p.slot_dep + __ldg(&p.ks[T.k].slot0);
    const uint64_t *oh = p.ohi + T.hi0, *ol = ROWS ? p.olo + __ldg(p.olo_off + T.m) : nullptr;
    const uint64_t ones = ROWS ? 0ull : (1ull << T.m) - 1;
    int64_t hi;
    int q, nc;
    if (!ROWS)
        for (int g = ptid; g < G; g += kPT) {
            win_unit(T, g, 0, p.co, &hi, &q, &nc);
            ncol[g] = (uint8_t)max(nc, 0);
        }
    win_unit(T, 0, 0, p.co, &hi, &q, &nc);
    const bool one = !ROWS && T.lone;  // every entry under the same o_hi word
    const uint64_t oh0 = nc > 0 ? __ldg(oh + hi) | ones : 0;
    for (int i0 = ptid; i0 < tot; i0 += U * kPT) {
        uint64_t word[U];
        int add[U];
#pragma unroll
        for (int v = 0; v < U; ++v) {
            const int i = i0 + v * kPT;
            word[v] = ~0ull;
            add[v] = 0;
            if (i >= tot) continue;
            const int e = ROWS ? i >> p.cos : per == 2 ? i >> 1 : i, jo = ROWS ? i & (p.co - 1) : 0;
            const int h = ROWS ? (per == 2 && jo >= cc ? 1 : 0) : per == 2 ? i & 1 : 0, lr = ROWS ? jo - h * cc : 0;
            int g = 0;
            uint64_t o = oh0;
            if (!one) {
                g = (int)win_div((uint32_t)e, inv);
                win_unit(T, g, h, p.co, &hi, &q, &nc);
                if (lr < nc) o = __ldg(oh + hi) | ones;
            }
            if (lr >= nc) continue;
            const uint64_t part = __ldg(parts + (e - g * n));
            if (ROWS) word[v] = part | o | __ldg(ol + q + lr);
            else if (part != ~0ull) word[v] = part | o;
            if (!ROWS) add[v] = one ? 0 : q;
        }
        int64_t off[U];
        uint32_t rk[U];
#pragma unroll
        for (int v = 0; v < U; ++v)
            if (word[v] != ~0ull) {
                off[v] = __ldg(p.hi_off + (word[v] >> p.L));
                rk[v] = __ldg(p.lo_rank + ((uint32_t)word[v] & p.lomask));
            }
#pragma unroll
        for (int v = 0; v < U; ++v) {
            const int i = i0 + v * kPT;
            if (i < tot) base[i] = word[v] != ~0ull ? (I)(off[v] + (int64_t)rk[v] + add[v]) : ~(I)0;
        }
    }
}

// Rows kind: blocks of RL rows (64 bytes of memory) and CL columns, neighbouring
// lanes on neighbouring rows.
// WIDE (eight FP32 vectors): blocks of eight rows, a lane's column its 16-byte
// chunk.
template <int VB, bool WIDE>
struct RowBlocks {
    static constexpr int CW = 64 / VB, CL = VB == 8 || WIDE ? 4 : 2, RL = 32 / CL, NC = WIDE ? 1 : CW / CL;
    int nrows, nrb, tot;
    __device__ __forceinline__ RowBlocks(const WinParams &p, const WinTile &T)
        : nrows(__ldg(&p.ks[T.k].nrows)), nrb((nrows + RL - 1) / RL), tot(T.G * nrb) {}
    // place of this lane's row of block rb: rinfo word (~0 for none) and unit
    __device__ __forceinline__ uint32_t row(const uint32_t *rinfo, int rb, int lane, int *g) const {
        int q = 0;
        while (rb >= (q + 1) * nrb) ++q;
        *g = q;
        const int r = (rb - q * nrb) * RL + (WIDE ? lane / CL : lane % RL);
        return rb < tot && r < nrows ? rinfo[r] : ~0u;
    }
};

// The flips of this lane's two rows (eight slots apart) for its 16 bytes of
// columns: a (set here).  tile: the unit's rows; c16: 16 times the chunk.
template <class Pol, bool ROWS, bool BOND>
__device__ __forceinline__ void row_flips(const unsigned char *tile, const uint2 *lp, uint32_t counts,
                                          const typename Pol::C *coef, int ng, uint32_t c16,
                                          typename Pol::Acc (&a)[2][16 / sizeof(typename Pol::V)]) {
    using V = typename Pol::V;
    using Acc = typename Pol::Acc;
    constexpr int VL = 16 / sizeof(V);
    union Q {
        int4 q;
        V v[VL];
    };
#pragma unroll
    for (int i = 0; i < VL; ++i) {
        Pol::zero(a[0][i]);
        Pol::zero(a[1][i]);
    }
    if (BOND) {
        const int n = (int)counts;
        auto load = [&](uint32_t e, Q &q, typename Pol::C &c) {
            const uint32_t s = e & 1023u;
            q.q = *(const int4 *)(tile + (win_row_off(ROWS, s) ^ c16));
            c = coef[e >> 10];
        };
        auto two = [&](Acc(&s)[VL], uint32_t e) {
            Q q0, q1;
            typename Pol::C k0, k1;
            load(e & 0xffffu, q0, k0);
            load(e >> 16, q1, k1);
#pragma unroll
            for (int i = 0; i < VL; ++i) Pol::fma(s[i], k0, q0.v[i]);
#pragma unroll
            for (int i = 0; i < VL; ++i) Pol::fma(s[i], k1, q1.v[i]);
        };
        auto single = [&](Acc(&s)[VL], uint32_t e) {
            Q q;
            typename Pol::C k;
            load(e & 0xffffu, q, k);
#pragma unroll
            for (int i = 0; i < VL; ++i) Pol::fma(s[i], k, q.v[i]);
        };
#pragma unroll 1
        for (int i = n >> 2; i > 0; --i, lp += kWinRows) {
            const uint2 e = lp[0], f = lp[8];
            two(a[0], e.x);
            two(a[1], f.x);
            two(a[0], e.y);
            two(a[1], f.y);
        }
        if (n & 3) {
            const uint2 e = lp[0], f = lp[8];
            if (n & 2) {
                two(a[0], e.x);
                two(a[1], f.x);
            }
            if (n & 1) {
                single(a[0], n & 2 ? e.y : e.x);
                single(a[1], n & 2 ? f.y : f.x);
            }
        }
    } else {
        const uint32_t cc = c16 | c16 << 16;
#pragma unroll 1
        for (int g = 0; g < ng; ++g, counts >>= 8) {
            const int n = (int)(counts & 255u);
            const typename Pol::C c = coef[g];
            Acc s[2][VL];
#pragma unroll
            for (int i = 0; i < VL; ++i) {
                Pol::zero(s[0][i]);
                Pol::zero(s[1][i]);
            }
            auto two = [&](uint32_t e, uint32_t f) {
                e ^= cc;
                f ^= cc;
                Q q0, q1, q2, q3;
                q0.q = *(const int4 *)(tile + (e & 0xffffu));
                q2.q = *(const int4 *)(tile + (f & 0xffffu));
                q1.q = *(const int4 *)(tile + (e >> 16));
                q3.q = *(const int4 *)(tile + (f >> 16));
#pragma unroll
                for (int k = 0; k < VL; ++k) Pol::list(s[0][k], c, q0.v[k], q1.v[k]);
#pragma unroll
                for (int k = 0; k < VL; ++k) Pol::list(s[1][k], c, q2.v[k], q3.v[k]);
            };
#pragma unroll 1
            for (int i = n >> 2; i > 0; --i, lp += kWinRows) {
                const uint2 e = lp[0], f = lp[8];
                two(e.x, f.x);
                two(e.y, f.y);
            }
            if (n & 3) {
                uint2 e = lp[0], f = lp[8];
                lp += kWinRows;
                if (n & 2) {
                    two(e.x, f.x);
                    e.x = e.y;
                    f.x = f.y;
                }
                if (n & 1) {
                    Q q0, q1;
                    q0.q = *(const int4 *)(tile + ((e.x ^ c16) & 0xffffu));
                    q1.q = *(const int4 *)(tile + ((f.x ^ c16) & 0xffffu));
#pragma unroll
                    for (int k = 0; k < VL; ++k) Pol::list(s[0][k], c, q0.v[k]);
#pragma unroll
                    for (int k = 0; k < VL; ++k) Pol::list(s[1][k], c, q1.v[k]);
                }
            }
#pragma unroll
            for (int k = 0; k < VL; ++k) {
                Pol::mul_add(a[0][k], c, s[0][k]);
                Pol::mul_add(a[1][k], c, s[1][k]);
            }
        }
    }
}

__device__ __forceinline__ void cp_async_v(void *dst, const void *src, int bytes) {
    const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
    if (bytes == 16) asm volatile("cp.async.cg.shared.global.L2::256B [%0], [%1], 16;\n" ::"r"(d), "l"(src));
    else if (bytes == 8) asm volatile("cp.async.ca.shared.global.L2::256B [%0], [%1], 8;\n" ::"r"(d), "l"(src));
    else asm volatile("cp.async.ca.shared.global.L2::256B [%0], [%1], 4;\n" ::"r"(d), "l"(src));
}
// Hardware barrier `id` of n threads: wait for all, or only be counted.
__device__ __forceinline__ void bar_sync(int id, int n) {
    __syncwarp();
    asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void bar_arrive(int id, int n) {
    __threadfence_block();
    __syncwarp();
    asm volatile("bar.arrive %0, %1;\n" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ void add4(PolF32::Acc (&a)[4], float4 v) {
    a[0].a += v.x;
    a[1].a += v.y;
    a[2].a += v.z;
    a[3].a += v.w;
}

template <class T>
__device__ __forceinline__ T shfl_xor(T v, int mask) {
    union {
        T v;
        int w[sizeof(T) / 4];
    } u;
    u.v = v;
#pragma unroll
    for (int i = 0; i < (int)(sizeof(T) / 4); ++i) u.w[i] = __shfl_xor_sync(0xffffffffu, u.w[i], mask);
    return u.v;
}

constexpr int kBarFull = 1, kBarEmpty = 3, kBarFlip = 5, kBarCopy = 6, kBarLook = 7;  // full and empty: + the tile's buffer

// A read of partial sums; the L2 fetches the 256 bytes around it, which the
// next tiles take.
template <class T>
__device__ __forceinline__ T ld_ahead(const T *p) {
    union {
        T v;
        unsigned long long w;
        unsigned h;
    } u;
    if constexpr (sizeof(T) == 8) asm volatile("ld.global.L2::256B.u64 %0, [%1];\n" : "=l"(u.w) : "l"(p) : "memory");
    else asm volatile("ld.global.L2::256B.u32 %0, [%1];\n" : "=r"(u.h) : "l"(p) : "memory");
    return u.v;
}
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.commit_group;\n" ::);
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
}

// Copies a tile in: the copying warps' part.
template <class Pol, bool ROWS, int NVS, typename I>
__device__ __forceinline__ void tile_in(const WinParams &p, const WinTile &T, const I *base, const uint8_t *ncol,
                                        unsigned char *tile, const typename Pol::V *x, int ptid) {
    using V = typename Pol::V;
    constexpr int VB = sizeof(V), VL = 16 / VB;
    constexpr bool WIDE = NVS == 3;
    const int lane = ptid & 31;
    for (int i = ptid; i < T.G * 8; i += kPT)  // the zero rows
        *(int4 *)(tile + ((i >> 3) * T.nslot + T.nslot - 2) * 64 + (i & 7) * 16) = make_int4(0, 0, 0, 0);
    if constexpr (ROWS) {
        using R = RowBlocks<VB, WIDE>;
        const R rows(p, T);
        const uint32_t *ri = p.rinfo + __ldg(&p.ks[T.k].row0);
        const int cl = WIDE ? lane & 3 : lane / R::RL, nwhi = T.nwhi, unit_bytes = T.nslot * 64;
        constexpr int U = 4;
        for (int rb = ptid >> 5; rb < rows.tot; rb += U * (kPT / 32)) {
            uint32_t e[U];
            int g[U];
#pragma unroll
            for (int u = 0; u < U; ++u) e[u] = rows.row(ri, rb + u * (kPT / 32), lane, &g[u]);
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (e[u] == ~0u) continue;
                const I *bw = base + ((g[u] * nwhi + ((e[u] >> 10) & 255u)) << p.cos);
                unsigned char *row = tile + g[u] * unit_bytes;
                const uint32_t ro = win_row_off(true, e[u] & 1023u);
#pragma unroll
                for (int cb = 0; cb < R::NC; ++cb) {
                    const int j = cb * R::CL + cl;
                    const I b = bw[WIDE ? j >> 1 : j];
                    if (b == ~(I)0) continue;
                    const int64_t q = (int64_t)b + (e[u] >> 18);
                    if constexpr (WIDE) cp_async_v(row + (ro ^ (uint32_t)j << 4), x + 8 * q + 4 * (j & 1), 16);
                    else cp_async_v(row + (ro ^ ((uint32_t)(j & 3) << 4 | (uint32_t)((j >> 2) * VB))), x + q, VB);
                }
            }
        }
    } else if constexpr (WIDE) {
        // four lanes to a row of two words o of eight values each
        const int c = ptid & 3, tot = T.G * kWinRows * T.nstep, cc = T.cc;
        const bool plain = T.per == 1;
        const int h = !plain && (c >> 1) >= cc ? 1 : 0, lr = (c >> 1) - h * cc;
        const float *xl = x + 8 * (int64_t)(T.q0 + lr) + 4 * (c & 1);
        unsigned char *dst = tile + (ptid >> 2) * 64 + (c << 4);
        for (int gs = ptid >> 2; gs < tot; gs += kPT / 4, dst += kPT * 16) {
            const int g = T.lone ? 0 : (int)win_div((uint32_t)gs, T.inv_unit);
            const int nc = T.lone ? T.nc0 : plain ? (int)ncol[g] : cc;
            const I b = base[plain ? gs : 2 * gs + h];
            if (b != ~(I)0 && lr < nc) cp_async_v(dst + g * 128, xl + 8 * (int64_t)b, 16);
        }
    } else {
        // eight lanes to a row, so that a warp access touches four 64-byte
        // runs of memory: the L1 tags, one 128-byte line a clock, are what
        // these accesses cost
        constexpr int NV = VL / 2;  // values of a lane and row
        const int j = ptid & 7, G = T.G, tot = G * kWinRows * T.nstep, cc = T.cc;
        const uint32_t inv = T.inv_unit;
        const bool plain = T.per == 1;
        int lr[NV], h[NV];
#pragma unroll
        for (int i = 0; i < NV; ++i) {
            const int jo = j + 8 * i;
            h[i] = !plain && jo >= cc ? 1 : 0;
            lr[i] = jo - h[i] * cc;
        }
        unsigned char *dst = tile + (ptid >> 3) * 64 + ((j & 3) << 4) + (j >> 2) * VB;
        if (T.lone) {
            const V *xl = x + T.q0 + lr[0];
            const bool in0 = lr[0] < T.nc0, in1 = NV > 1 && lr[NV - 1] < T.nc0;
            constexpr int U = 8;
            for (int gs = ptid >> 3; gs < tot; gs += U * (kPT / 8), dst += U * kPT * 8) {
                I b[U];
#pragma unroll
                for (int u = 0; u < U; ++u) b[u] = gs + u * (kPT / 8) < tot ? base[gs + u * (kPT / 8)] : ~(I)0;
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    if (b[u] == ~(I)0) continue;
                    const V *src = xl + b[u];
                    if (in0) cp_async_v(dst + u * kPT * 8, src, VB);
                    if (NV > 1 && in1) cp_async_v(dst + u * kPT * 8 + 2 * VB, src + 8, VB);
                }
            }
        } else {
            for (int gs = ptid >> 3; gs < tot; gs += kPT / 8, dst += kPT * 8) {
                const int g = (int)win_div((uint32_t)gs, inv), nc = plain ? (int)ncol[g] : cc;
#pragma unroll
                for (int i = 0; i < NV; ++i) {
                    const I b = base[plain ? gs : 2 * gs + h[i]];
                    if (b != ~(I)0 && lr[i] < nc)
                        cp_async_v(dst + g * 128 + i * 2 * VB, x + ((int64_t)b + lr[i]), VB);
                }
            }
        }
    }
}

// One pass, one CTA per SM.  It walks the tiles of its runs (win_divide; popcount
// by popcount, so the lists are loaded once per run) in three roles: one warp plans
// (win_next: the shape of tile i + 2), six look up row offsets (tile i + 1) and copy
// (tile i), seventeen flip, a step being sixteen rows, two to each four lanes.
//
// What may be written again, and what allows it: a tile's buffer (two, by i & 1)
// once the flipping warps have arrived at kBarEmpty of tile i - 2, for which the
// copying warps wait before tile i; the ring's shapes (four, by i & 3), written by
// the planning warp for tile i + 2 after kBarCopy of tile i, which the copying warps
// reach only then, so that tile i - 2 is done with; row offsets and ncols (three or
// two sets, and four, by the number of their last change, gen), written for tile
// i + 1 while tiles i and i - 1 are read, or with two sets for tile i before it is
// copied.  The flipping warps take tile i after kBarFull, for which the copying
// warps arrive when their copies are there; the lists and the rows kind's sums in
// the tile's place go between two kBarFlip of the flipping warps alone.  All roles
// walk the same tiles, so every wait has its arrivals.
//
// Columns kind: a step reads the row's earlier sums (acc, y's own memory)
// before its flips and writes the new ones after them, 32 bytes per row and
// access.  Rows kind: memory runs along the rows, whose order the steps do not
// follow, so the sums stay in registers until no row reads the tile any more,
// go into the tile's place and out from there.  I: uint32 row offsets below 2^32
// rows.
template <class Pol, bool ROWS, bool BOND, int NVS, typename I>
__device__ __forceinline__ void win_pass(const WinParams &p, const typename Pol::V *__restrict__ x,
                                         typename Pol::Acc *acc, typename Pol::Y *y) {
    using V = typename Pol::V;
    using C = typename Pol::C;
    using D = typename Pol::D;
    using Acc = typename Pol::Acc;
    constexpr int VB = sizeof(V), VL = 16 / VB;
    constexpr bool WIDE = NVS == 3;
    static_assert(NVS == 0 || (WIDE && VB == 4), "one vector, or eight in FP32");
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ uint8_t ncols[4][64];
    __shared__ WinTile ring[4];  // by tile number
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    C *coef = (C *)(smem + p.sm_coef);
    for (int i = tid; i < p.ncoef; i += kT) coef[i] = ((const C *)p.coef[Pol::kArith])[i];
    const int ntiles = __ldg(&p.ctas[blockIdx.x].ntiles);
    if (ntiles <= 0) return;
    __syncthreads();
    if (warp >= kCW) {
        // Tile i is copied as soon as tile i - 2 is done with; while its data
        // are on their way, the row offsets of tile i + 1 and the shape of
        // tile i + 2 (by the planning warp) are looked up.
        const int ptid = tid - 32 * kCW;
        const bool ahead = p.nbase_bufs == 3;
        auto base_of = [&](const WinTile &T) { return (I *)(smem + p.sm_base + (ahead ? T.gen % 3 : T.gen & 1) * p.base_bytes); };
        auto look_up = [&](int i) {
            const WinTile &T = ring[i & 3];
            if (T.fresh) tile_base<ROWS, I>(p, T, base_of(T), ncols[T.gen & 3], ptid);
        };
        if (ptid >= kPT) {  // the planning warp
            WinTile w;
            w.seg = 0;
            w.gen = -1;
            w.uh = 0;
            w.lone = 0;
            WinWalk walk{__ldg(&p.ctas[blockIdx.x].run0), 0, 0};
            auto shape = [&](int i) {  // one thread: the shape of tile i
                if (i < ntiles) {
                    win_next(p.runs, p.segs, p.nseg, p.ks, ROWS, p.co, &walk, &w);
                    ring[i & 3] = w;
                }
            };
            if (ptid == kPT) {
                shape(0);
                shape(1);
            }
            bar_sync(kBarCopy, kPT + 32);
            for (int i = 0; i < ntiles; ++i) {
                bar_sync(kBarCopy, kPT + 32);  // tile i - 2 is done with
                if (ptid == kPT) shape(i + 2);
            }
            return;
        }
        bar_sync(kBarCopy, kPT + 32);
        if (ahead) look_up(0);
        for (int i = 0; i < ntiles; ++i) {
            if (i >= 2) bar_sync(kBarEmpty + (i & 1), kMeet);
            if (!ahead) {
                look_up(i);
                bar_sync(kBarLook, kPT);
            }
            bar_sync(kBarCopy, kPT + 32);  // this tile's row offsets and the next one's shape are there
            const WinTile &T = ring[i & 3];
            tile_in<Pol, ROWS, NVS, I>(p, T, base_of(T), ncols[T.gen & 3], smem + (i & 1) * p.sm_tile1, x, ptid);
            if (ahead && i + 1 < ntiles) look_up(i + 1);
            cp_async_wait();
            bar_arrive(kBarFull + (i & 1), kMeet);
        }
        return;
    }
    uint32_t *list = (uint32_t *)(smem + p.sm_list);
    uint2 *steps = (uint2 *)(smem + p.sm_step);
    uint32_t *rinfo = (uint32_t *)(smem + p.sm_rinfo);  // rows kind
    const uint32_t c16 = (uint32_t)(lane & 3) << 4;
    const typename Pol::Out oset = Pol::out_setup(p, Pol::kArith < 2 ? __ldg(p.state) : 0);
    int cur = -1, off = 0;  // off: where the deal of steps to warps stands
    const D *diag = nullptr;
    auto lists = [&](int k) {  // the flip lists (and, rows kind, the rows) of popcount k
        cur = k;
        const WinK &K = p.ks[k];
        const int4 *gl = (const int4 *)(p.list + __ldg(&K.list0));
        const uint2 *go = p.step + __ldg(&K.step0);
        const int nl = __ldg(&K.nlist) / 4, ns = __ldg(&K.nstep);
#pragma unroll 4
        for (int q = tid; q < nl; q += 32 * kCW) ((int4 *)list)[q] = __ldg(gl + q);
        for (int q = tid; q < ns; q += 32 * kCW) steps[q] = __ldg(go + q);
        if (ROWS) {
            const int nr = __ldg(&K.nrows);
            const uint32_t *gr = p.rinfo + __ldg(&K.row0);
            for (int q = tid; q < nr; q += 32 * kCW) rinfo[q] = __ldg(gr + q);
        }
        diag = (const D *)p.diag[Pol::kArith] + __ldg(&K.slot0);
    };
    lists(__ldg(&p.ctas[blockIdx.x].k0));  // while the first tile is copied
    bar_sync(kBarFlip, 32 * kCW);
    for (int i = 0; i < ntiles; ++i) {
        bar_sync(kBarFull + (i & 1), kMeet);
        const WinTile &T = ring[i & 3];
        const int nstep = T.nstep, ntot = T.G * nstep, unit_bytes = T.nslot * 64;
        const uint32_t inv_step = T.inv_step;
        unsigned char *tile = smem + (i & 1) * p.sm_tile1;
        const I *base = (const I *)(smem + p.sm_base + (p.nbase_bufs == 3 ? T.gen % 3 : T.gen & 1) * p.base_bytes);
        const uint8_t *ncol = ncols[T.gen & 3];
        if (T.k != cur) {
            bar_sync(kBarFlip, 32 * kCW);
            lists(T.k);
            bar_sync(kBarFlip, 32 * kCW);
        }
        auto step = [&](int o, Acc(&a)[2][VL]) {  // the sums of step o's rows
            const int g = (int)win_div((uint32_t)o, inv_step), oo = o - g * nstep;
            const unsigned char *unit = tile + g * unit_bytes;
            const uint2 hd = steps[oo];
            const uint32_t slot = (uint32_t)(kWinRows * oo + (lane >> 2));
            const D d0 = __ldg(diag + slot), d1 = __ldg(diag + slot + 8);
            row_flips<Pol, ROWS, BOND>(unit, (const uint2 *)list + hd.x * kWinRows + (lane >> 2), hd.y, coef, p.ng, c16, a);
            union {
                int4 q;
                V v[VL];
            } x0, x1;
            x0.q = *(const int4 *)(unit + (win_row_off(ROWS, slot) ^ c16));
            x1.q = *(const int4 *)(unit + (win_row_off(ROWS, slot + 8) ^ c16));
#pragma unroll
            for (int k = 0; k < VL; ++k) {
                Pol::diag(a[0][k], d0, x0.v[k]);
                Pol::diag(a[1][k], d1, x1.v[k]);
            }
        };
        // steps are dealt to the warps in turn across tiles
        int o0 = warp - off;
        if (o0 < 0) o0 += kCW;
        off = (off + ntot) % kCW;
        if constexpr (!ROWS && WIDE) {
            const bool plain = T.per == 1, many = plain && !T.lone;
            const int c = lane & 3, cc = T.cc, cols = plain ? T.nc0 : cc;
            const int h = !plain && (c >> 1) >= cc ? 1 : 0, lr = (c >> 1) - h * cc;
            const int64_t shift = 8 * (int64_t)(T.q0 + lr) + 4 * (c & 1);
            for (int o = o0; o < ntot; o += kCW) {
                Acc a[2][VL];
                float4 prev[2];
                float *at[2];
                const int nc = many ? (int)ncol[win_div((uint32_t)o, inv_step)] : cols;
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    const int row = kWinRows * o + (lane >> 2) + 8 * u;
                    const I b = base[plain ? row : 2 * row + h];
                    at[u] = b != ~(I)0 && lr < nc ? (float *)y + 8 * (int64_t)b + shift : nullptr;
                    if (!p.first && at[u]) prev[u] = *(const float4 *)at[u];
                }
                step(o, a);
#pragma unroll
                for (int u = 0; u < 2; ++u)
                    if (at[u]) {
                        if (!p.first) add4(a[u], prev[u]);
                        *(float4 *)at[u] = make_float4(a[u][0].a, a[u][1].a, a[u][2].a, a[u][3].a);
                    }
            }
        } else if constexpr (!ROWS) {
            // After its flips a lane trades half of its columns with the lane
            // four on, which has the neighbouring row: then eight lanes hold a
            // row's values and an access touches four 64-byte runs of memory
            // (as in tile_in).  The earlier sums are read in that order before
            // the flips.
            constexpr int NV = VL / 2;
            const bool plain = T.per == 1, many = plain && !T.lone;
            const int cc = T.cc, cols = plain ? T.nc0 : cc, odd = (lane >> 2) & 1, q0 = T.q0;
            for (int o = o0; o < ntot; o += kCW) {
                Acc a[2][VL], prev[2][2][NV];
                const int gs = kWinRows * o + ((lane >> 2) & ~1);
                const int nc = many ? (int)ncol[win_div((uint32_t)o, inv_step)] : cols;
                // value i of row e of the pair eight u slots on: its index, or false
                auto place = [&](int u, int e, int i, int64_t *q) -> bool {
                    const int jo = (lane & 3) + 4 * odd + 8 * i, h = !plain && jo >= cc ? 1 : 0;
                    const int lr = jo - (h ? cc : 0), row = gs + 8 * u + e;
                    const I b = base[plain ? row : 2 * row + h];
                    *q = (int64_t)(I)(b + (I)(q0 + lr));
                    return b != ~(I)0 && lr < nc;
                };
                if (!p.first)
#pragma unroll
                    for (int u = 0; u < 2; ++u)
#pragma unroll
                        for (int e = 0; e < 2; ++e)
#pragma unroll
                            for (int i = 0; i < NV; ++i) {
                                int64_t q;
                                if (place(u, e, i, &q)) prev[u][e][i] = ld_ahead(acc + q);
                            }
                step(o, a);
#pragma unroll
                for (int u = 0; u < 2; ++u) {
                    Acc v[2][NV];
#pragma unroll
                    for (int i = 0; i < NV; ++i) {
                        const Acc give = odd ? a[u][2 * i] : a[u][2 * i + 1], keep = odd ? a[u][2 * i + 1] : a[u][2 * i];
                        const Acc got = shfl_xor(give, 4);
                        v[0][i] = odd ? got : keep;
                        v[1][i] = odd ? keep : got;
                    }
#pragma unroll
                    for (int e = 0; e < 2; ++e)
#pragma unroll
                        for (int i = 0; i < NV; ++i) {
                            int64_t q;
                            if (!place(u, e, i, &q)) continue;
                            Acc s = v[e][i];
                            if (!p.first) Pol::merge(s, prev[u][e][i]);
                            if (p.last) y[q] = Pol::result(s, oset);
                            else acc[q] = s;
                        }
                }
            }
        } else {
            Acc held[kSteps][2][VL];
#pragma unroll
            for (int s = 0; s < kSteps; ++s)
                if (o0 + s * kCW < ntot) step(o0 + s * kCW, held[s]);
            bar_sync(kBarFlip, 32 * kCW);
#pragma unroll
            for (int s = 0; s < kSteps; ++s) {
                const int o = o0 + s * kCW;
                if (o < ntot) {
                    const int g = (int)win_div((uint32_t)o, inv_step);
                    const uint32_t slot = (uint32_t)(kWinRows * (o - g * nstep) + (lane >> 2));
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        union {
                            int4 q;
                            Acc v[VL];
                        } w;
#pragma unroll
                        for (int k = 0; k < VL; ++k) w.v[k] = held[s][u][k];
                        *(int4 *)(tile + g * unit_bytes + (win_row_off(true, slot + 8 * u) ^ c16)) = w.q;
                    }
                }
            }
            bar_sync(kBarFlip, 32 * kCW);
            // out: the earlier sums of U blocks of rows are read together
            using R = RowBlocks<VB, WIDE>;
            const R rows(p, T);
            const int cl = WIDE ? lane & 3 : lane / R::RL, nwhi = T.nwhi;
            if constexpr (WIDE) {
                constexpr int U = 4;
                for (int rb = warp; rb < rows.tot; rb += U * kCW) {
                    float *at[U];
                    float4 prev[U];
                    uint32_t from[U];
#pragma unroll
                    for (int u = 0; u < U; ++u) {
                        int g = 0;
                        const uint32_t e = rb + u * kCW < rows.tot ? rows.row(rinfo, rb + u * kCW, lane, &g) : ~0u;
                        from[u] = (uint32_t)(g * unit_bytes) + (win_row_off(true, e & 1023u) ^ c16);
                        const I b = e != ~0u ? base[((g * nwhi + ((e >> 10) & 255u)) << p.cos) + (cl >> 1)] : ~(I)0;
                        at[u] = b != ~(I)0 ? (float *)y + 8 * ((int64_t)b + (e >> 18)) + 4 * (cl & 1) : nullptr;
                        if (!p.first && at[u]) prev[u] = *(const float4 *)at[u];
                    }
#pragma unroll
                    for (int u = 0; u < U; ++u)
                        if (at[u]) {
                            float4 v = *(const float4 *)(tile + from[u]);
                            if (!p.first) {
                                v.x += prev[u].x;
                                v.y += prev[u].y;
                                v.z += prev[u].z;
                                v.w += prev[u].w;
                            }
                            *(float4 *)at[u] = v;
                        }
                }
            } else {
            constexpr int U = VB == 8 ? 4 : 2;
            for (int rb = warp; rb < rows.tot; rb += U * kCW) {
                uint32_t row[U];
                I idx[U][R::NC];
                Acc prev[U][R::NC];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    int g;
                    const uint32_t e = rb + u * kCW < rows.tot ? rows.row(rinfo, rb + u * kCW, lane, &g) : (g = 0, ~0u);
                    row[u] = (uint32_t)(g * unit_bytes) + win_row_off(true, e & 1023u);
                    const I *bw = base + ((g * nwhi + ((e >> 10) & 255u)) << p.cos);
#pragma unroll
                    for (int cb = 0; cb < R::NC; ++cb) {
                        const int j = cb * R::CL + cl;
                        const I b = e != ~0u ? bw[j] : ~(I)0;
                        idx[u][cb] = b != ~(I)0 ? b + (I)(e >> 18) : b;
                        if (!p.first && b != ~(I)0) prev[u][cb] = ld_ahead(acc + idx[u][cb]);
                    }
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
#pragma unroll
                    for (int cb = 0; cb < R::NC; ++cb)
                        if (idx[u][cb] != ~(I)0) {
                            const int j = cb * R::CL + cl;
                            const int64_t q = (int64_t)idx[u][cb];
                            Acc a = *(const Acc *)(tile + (row[u] ^ ((uint32_t)(j & 3) << 4 | (uint32_t)((j >> 2) * VB))));
                            if (!p.first) Pol::merge(a, prev[u][cb]);
                            if (p.last) y[q] = Pol::result(a, oset);
                            else acc[q] = a;
                        }
            }
            }
        }
        if (i + 2 < ntiles) bar_arrive(kBarEmpty + (i & 1), kMeet);
    }
}

// FP64: in the arithmetic that k_x64_convert chose.  FP32: in FP32.
template <bool F64, bool ROWS, bool BOND, int NVS, typename I>
__global__ void __launch_bounds__(kT, 1) k_win(const __grid_constant__ WinParams p, const void *__restrict__ x, void *y) {
    if constexpr (F64) {
        if (__ldg(p.state + 1))
            win_pass<PolFX, ROWS, BOND, NVS, I>(p, (const long long *)x, (PolFX::Acc *)y, (double *)y);
        else
            win_pass<PolDF, ROWS, BOND, NVS, I>(p, (const float2 *)x, (PolDF::Acc *)y, (double *)y);
    } else {
        win_pass<PolF32, ROWS, BOND, NVS, I>(p, (const float *)x, (PolF32::Acc *)y, (float *)y);
    }
}

}  // namespace

// ------------------------------------------------------------ host side

// Tables gathered on the host for one allocation and one copy.
struct Pack {
    std::vector<unsigned char> bytes;
    std::vector<std::pair<void **, size_t>> at;
    template <typename E>
    void add(E **dst, const std::vector<E> &v) {
        const size_t o = (bytes.size() + 15) / 16 * 16;
        bytes.resize(o + std::max<size_t>(1, v.size()) * sizeof(E));
        if (!v.empty()) memcpy(&bytes[o], v.data(), v.size() * sizeof(E));
        at.push_back({(void **)dst, o});
    }
    xd_status upload(unsigned char **buf) {
        XD_CUDA(dev_malloc((void **)buf, bytes.size()));
        XD_CUDA(cudaMemcpy(*buf, bytes.data(), bytes.size(), cudaMemcpyHostToDevice));
        for (auto &p : at) *p.first = *buf + p.second;
        return XD_OK;
    }
};

bool win_layout_wanted(const xd_basis_s *b) { return large_block(b); }

// The passes of the block's graph, the words outside their windows and the
// tiles; the flip lists follow with the couplings (win_ham_tables).
xd_status win_layout_build(xd_basis_s *b) {
    WinLayoutHost &wl = b->win;
    grid_for(1, 1, 1);
    wl.pairs = win_pairs((const int32_t *)b->bonds.data(), b->nb, &wl.pair_of);
    std::vector<WinPlan> plan = win_plan(b->N, b->nup, wl.pairs, g_num_sms);
    wl.pass.resize(plan.size());
    Pack pack;
    for (size_t ip = 0; ip < plan.size(); ++ip) {
        WinPlan &s = plan[ip];
        WinPassDev &d = wl.pass[ip];
        d.p = s.p;
        pack.add(&d.d_ohi, s.T.ohi);
        pack.add(&d.d_olo, s.T.olo);
        pack.add(&d.d_olo_off, s.T.olo_off);
        pack.add(&d.d_whi, s.T.whi);
        s.T.ohi = s.T.olo = std::vector<uint64_t>();  // up to a hundred MB at 40 sites
        for (int q = 0; q < kWinForms; ++q) {
            d.nseg[q] = (int)s.segs[q].size();
            d.nctas[q] = (int)s.ctas[q].size() - 1;
            d.nbase[q] = s.nbase[q];
            pack.add(&d.d_segs[q], s.segs[q]);
            pack.add(&d.d_ctas[q], s.ctas[q]);
            pack.add(&d.d_runs[q], s.runs[q]);
        }
    }
    XD_TRY(pack.upload(&wl.buf));
    wl.spmm32 = spmm_better(b, plan, false);
    wl.spmm8 = spmm_better(b, plan, true);
    wl.ok = true;
    return XD_OK;
}

void win_layout_free(xd_basis_s *b) {
    cudaFree(b->win.buf);
    b->win = WinLayoutHost();
}

// The couplings of the distinct pairs.
static std::vector<double> pair_couplings(const xd_basis_s *b, const double *J) {
    std::vector<double> Jp(b->win.pairs.size(), 0.0);
    for (int t = 0; t < b->nb; ++t) Jp[b->win.pair_of[t]] += J[t];
    return Jp;
}

// Flip lists of the passes whose pattern of equal couplings is another than the
// handle's, in new allocations (out[pass].buf; null: the handle's lists stay).
// Flips are listed coupling by coupling when a pass has at most kWinMaxGroups of
// them (one multiplication per row and coupling; measured at the 4x8 J1-J2
// lattice against entries that carry their bond) and they fit
// (win_fitting_lists), else with the bond in each entry.  Nothing of the handle
// changes, so that an allocation that fails leaves it as it was; the caller frees
// what is left in `out`.
xd_status win_ham_lists(const xd_ham_s *h, const double *J, std::vector<WinPassHam> *out) {
    const xd_basis_s *b = h->b;
    const WinLayoutHost &wl = b->win;
    const std::vector<double> Jp = pair_couplings(b, J);
    const bool wide = win_wide(b->dim_u1);
    out->assign(wl.pass.size(), WinPassHam());
    for (size_t ip = 0; ip < wl.pass.size(); ++ip) {
        const WinPassDev &pd = wl.pass[ip];
        const WinPass &p = pd.p;
        std::vector<double> vals;
        std::vector<int> gid(p.bonds.size());
        for (size_t t = 0; t < gid.size(); ++t) {
            const double v = Jp[p.bonds[t]];
            gid[t] = (int)(std::find(vals.begin(), vals.end(), v) - vals.begin());
            if (gid[t] == (int)vals.size()) vals.push_back(v);
        }
        const int groups = (int)vals.size() <= kWinMaxGroups ? (int)vals.size() : 0;
        if (!groups) std::fill(gid.begin(), gid.end(), 0);
        if (ip < h->win.size() && h->win[ip].groups == groups && h->win[ip].gid == gid) continue;
        WinPassHam &w = (*out)[ip];
        WinTables T;
        w.ng = win_fitting_lists(p, wl.pairs, pd.nbase, wide, gid, groups, &T, w.fit);
        w.ncoef = w.ng ? w.ng : kWinMaxBonds + 1;
        w.groups = groups;
        w.gid = gid;
        w.slot_word = T.slot_word;
        w.maxslots = T.maxslots;
        w.maxlist = T.maxlist;
        w.maxstep = T.maxstep;
        const size_t nslot = T.slot_word.size();
        auto take = [&](size_t bytes) {
            const size_t at = w.bytes;
            w.bytes += (bytes + 15) / 16 * 16;
            return at;
        };
        w.oks = take(T.k.size() * sizeof(WinK));
        w.osd = take(nslot * 8);
        w.ori = take(T.rinfo.size() * 4);
        w.oli = take(T.list.size() * 4);
        w.ost = take(T.step.size() * 4);
        w.ovar = w.bytes;
        const size_t cs[3] = {8, 4, 4};
        for (int a = 0; a < 3; ++a) {
            w.oc[a] = take((kWinMaxBonds + 1) * cs[a]);
            w.od[a] = take(nslot * cs[a]);
        }
        std::vector<unsigned char> host(w.ovar, 0);
        memcpy(&host[w.oks], T.k.data(), T.k.size() * sizeof(WinK));
        memcpy(&host[w.osd], T.slot_dep.data(), nslot * 8);
        memcpy(&host[w.ori], T.rinfo.data(), T.rinfo.size() * 4);
        memcpy(&host[w.oli], T.list.data(), T.list.size() * 4);
        memcpy(&host[w.ost], T.step.data(), T.step.size() * 4);
        cudaError_t e = dev_malloc((void **)&w.buf, w.bytes);
        if (e == cudaSuccess) e = cudaMemcpy(w.buf, host.data(), w.ovar, cudaMemcpyHostToDevice);
        if (e != cudaSuccess) return cuda_status(e, "window lists");
    }
    return XD_OK;
}

// The lists of win_ham_lists, and the coefficients and diagonals of every pass
// for the handle's couplings.
xd_status win_ham_tables(xd_ham_s *h, std::vector<WinPassHam> *lists) {
    const xd_basis_s *b = h->b;
    const WinLayoutHost &wl = b->win;
    const int np = (int)wl.pairs.size();
    h->win.resize(wl.pass.size());
    // products in flight on any stream read the lists that go
    bool replaced = false;
    for (size_t ip = 0; ip < lists->size(); ++ip) replaced = replaced || (h->win[ip].buf && (*lists)[ip].buf);
    if (replaced) XD_CUDA(cudaDeviceSynchronize());
    std::fill(h->win_fit, h->win_fit + kWinForms, true);
    for (size_t ip = 0; ip < lists->size(); ++ip) {
        WinPassHam &w = h->win[ip];
        if ((*lists)[ip].buf) {
            cudaFree(w.buf);
            w = (*lists)[ip];
            (*lists)[ip].buf = nullptr;
        }
        for (int f = 0; f < kWinForms; ++f) h->win_fit[f] = h->win_fit[f] && w.fit[f];
    }
    double q = 1.0;
    std::vector<int> k;
    h->x64_fx_ok = find_quantum(h->J, &q, &k);
    const std::vector<double> Jp = pair_couplings(b, h->J.data());
    std::vector<int> kp(np, 0);
    int64_t kabs = 0;
    for (int t = 0; t < b->nb && h->x64_fx_ok; ++t) {
        kp[wl.pair_of[t]] += k[t];
        kabs += std::abs(k[t]);
    }
    // every partial sum is at most 3 sum|k_b| max|X| < 2^62
    int lg = 0;
    while ((int64_t(1) << lg) < 3 * std::max<int64_t>(1, kabs)) ++lg;
    h->x64_B = 62 - lg;
    h->x64_qs = 0.25 * q;
    for (size_t ip = 0; ip < wl.pass.size(); ++ip) {
        const WinPassHam &w = h->win[ip];
        const WinPass &p = wl.pass[ip].p;
        const int nwb = (int)p.bonds.size(), ws = (int)p.S.size();
        // coefficients (double-float, fixed point, FP32) and the window words' diagonals
        auto pair = [](double d) {
            const float c = (float)d;
            return make_float2(c, (float)(d - (double)c));
        };
        std::vector<unsigned char> var(w.bytes - w.ovar, 0);
        float2 *c0 = (float2 *)&var[w.oc[0] - w.ovar], *d0 = (float2 *)&var[w.od[0] - w.ovar];
        int *c1 = (int *)&var[w.oc[1] - w.ovar], *d1 = (int *)&var[w.od[1] - w.ovar];
        float *c2 = (float *)&var[w.oc[2] - w.ovar], *d2 = (float *)&var[w.od[2] - w.ovar];
        std::vector<double> Dj(1u << ws, 0.0);
        std::vector<int> Dk(1u << ws, 0);
        for (int t = 0; t < nwb; ++t) {
            const auto &pr = wl.pairs[p.bonds[t]];
            const int at = w.ng ? w.gid[t] : t, kb = kp[p.bonds[t]];
            const double j = Jp[p.bonds[t]];
            c0[at] = pair(0.5 * j);
            c1[at] = 2 * kb;
            c2[at] = (float)(0.5 * j);
            int i0 = 0, i1 = 0;
            for (int i = 0; i < ws; ++i) {
                if (p.S[i] == pr.first) i0 = i;
                if (p.S[i] == pr.second) i1 = i;
            }
            for (uint32_t v = 0; v < (1u << ws); ++v) {
                const int s = 1 - 2 * (int)(((v >> i0) ^ (v >> i1)) & 1u);
                Dj[v] += s * 0.25 * j;
                Dk[v] += s * kb;
            }
        }
        for (size_t s = 0; s < w.slot_word.size(); ++s) {
            const uint32_t v = w.slot_word[s];
            if (v == 0xffffu) continue;
            d0[s] = pair(Dj[v]);
            d1[s] = Dk[v];
            d2[s] = (float)Dj[v];
        }
        XD_CUDA(cudaMemcpy(w.buf + w.ovar, var.data(), var.size(), cudaMemcpyHostToDevice));
    }
    return XD_OK;
}

void win_ham_free(xd_ham_s *h) {
    for (WinPassHam &w : h->win) cudaFree(w.buf);
    h->win.clear();
}

// The FP64 workspace (8 bytes per row, the two state words and the partials
// of the statistics pass) is allocated on first use.  When it does not fit,
// the call returns XD_ENOMEM and this product takes the FP64 block kernel;
// the next product tries again (the drivers that hold several vectors
// release the workspace when their own vectors do not fit, x64_release).
xd_status x64_workspace(xd_ham_s *h, int64_t dim) {
    grid_for(1, 1, 1);
    if (!h->d_x64_state) {
        cudaError_t e = dev_malloc((void **)&h->d_x64_state, 16 + (size_t)g_num_sms * kStatPerSm * sizeof(ExpSum));
        if (e != cudaSuccess) {
            cudaGetLastError();
            return XD_ENOMEM;
        }
    }
    if (h->d_x64_x) return XD_OK;
    cudaError_t e = dev_malloc((void **)&h->d_x64_x, (size_t)dim * 8);
    if (e != cudaSuccess) {
        cudaGetLastError();
        h->d_x64_x = nullptr;
        return XD_ENOMEM;
    }
    return XD_OK;
}

void x64_release(xd_ham_s *h) {
    if (h->d_x64_x) {
        lanczos_forget(h, false);  // captured Lanczos steps read the workspace
        cudaFree(h->d_x64_x);
        h->d_x64_x = nullptr;
    }
}

// The passes (win_fit is set); NVS = log2 of the vectors per row: 0, or 3 in FP32.
template <bool F64, int NVS>
static xd_status launch_passes(const xd_ham_s *h, const void *x, void *y, cudaStream_t st) {
    const xd_basis_s *b = h->b;
    const WinLayoutHost &wl = b->win;
    constexpr WinForm form = F64 ? kWinF64 : NVS ? kWinF32x8 : kWinF32;
    constexpr int co = kWinCols[form];
    static_assert(co == (64 / (F64 ? 8 : 4)) >> NVS, "64 bytes to a row of a tile");
    int cos = 0;
    while ((1 << cos) < co) ++cos;
    const bool wide = win_wide(b->dim_u1);
    for (size_t ip = 0; ip < wl.pass.size(); ++ip) {
        const WinPassDev &d = wl.pass[ip];
        const WinPassHam &w = h->win[ip];
        WinParams p;
        p.hi_off = b->d_hi_off;
        p.lo_rank = b->d_lo_rank;
        p.L = b->L;
        p.lomask = (uint32_t)((1ull << b->L) - 1);
        p.ks = (const WinK *)(w.buf + w.oks);
        p.segs = d.d_segs[form];
        p.nseg = d.nseg[form];
        p.ctas = d.d_ctas[form];
        p.runs = d.d_runs[form];
        p.c0 = d.p.c0;
        p.co = co;
        p.cos = cos;
        p.slot_dep = (const uint64_t *)(w.buf + w.osd);
        p.ohi = d.d_ohi;
        p.olo = d.d_olo;
        p.olo_off = d.d_olo_off;
        p.whi = d.d_whi;
        p.rinfo = (const uint32_t *)(w.buf + w.ori);
        p.list = (const uint32_t *)(w.buf + w.oli);
        p.step = (const uint2 *)(w.buf + w.ost);
        for (int q = 0; q < 3; ++q) {
            p.coef[q] = w.buf + w.oc[q];
            p.diag[q] = w.buf + w.od[q];
        }
        p.ncoef = w.ncoef;
        p.ng = w.ng;
        p.first = ip == 0;
        p.last = ip + 1 == wl.pass.size();
        p.qs = h->x64_qs;
        p.B = h->x64_B;
        p.state = h->d_x64_state;
        const WinSmem sm = win_smem(d.p.rows, w.maxslots, w.maxlist, w.maxstep, w.ncoef, d.nbase[form], wide);
        p.sm_tile1 = sm.tile1;
        p.sm_list = sm.list;
        p.sm_step = sm.step;
        p.sm_coef = sm.coef;
        p.sm_rinfo = sm.rinfo;
        p.base_bytes = sm.base_bytes;
        p.nbase_bufs = sm.base_sets;
        p.sm_base = sm.base;
        auto go = [&](auto kern) -> xd_status {
            // the limit, not this pass's size: another thread may be about to launch a larger one
            XD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kWinSmem));
            const int grid = d.nctas[form];
            kern<<<grid, kT, sm.total, st>>>(p, x, y);
            XD_CUDA(cudaGetLastError());
            return XD_OK;
        };
        auto pick = [&](auto idx) -> xd_status {
            using I = decltype(idx);
            if (d.p.rows) return p.ng ? go(k_win<F64, true, false, NVS, I>) : go(k_win<F64, true, true, NVS, I>);
            return p.ng ? go(k_win<F64, false, false, NVS, I>) : go(k_win<F64, false, true, NVS, I>);
        };
        if constexpr (NVS == 0) XD_TRY(wide ? pick((unsigned long long)0) : pick((unsigned)0));
        else XD_TRY(pick((unsigned)0));  // win8_usable: no 64-bit row offsets
    }
    return XD_OK;
}

// Statistics of x, the choice of arithmetic and the conversion on the device,
// where the passes read the choice (no host synchronisation).
xd_status win_apply_f64(const xd_ham_s *h, const void *x, void *y, cudaStream_t st) {
    xd_ham_s *hm = const_cast<xd_ham_s *>(h);
    const int64_t dim = h->b->dim;
    XD_TRY(x64_workspace(hm, dim));
    x64_convert(h, x, dim, st);
    XD_CUDA(cudaGetLastError());
    return launch_passes<true, 0>(h, h->d_x64_x, y, st);
}

xd_status win_apply_f32(const xd_ham_s *h, const void *x, void *y, cudaStream_t st) {
    return launch_passes<false, 0>(h, x, y, st);
}

// Eight FP32 vectors: where these passes are estimated faster than the prefix
// blocks of xd_u1_spmm8.cu (spmm_better) and their tables fit (no 64-bit row
// offsets).
bool win8_usable(const xd_ham_s *h, const void *x, const void *y) {
    return h->win_fit[kWinF32x8] && !h->b->win.spmm8 && (((uintptr_t)x | (uintptr_t)y) & 15) == 0;
}

xd_status win8_apply(const xd_ham_s *h, const void *x, void *y, cudaStream_t st) {
    return launch_passes<false, 3>(h, x, y, st);
}

}  // namespace xd
