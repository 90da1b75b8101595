// xd_u1_rows.cuh -- the row loop of the plain U(1) product (pull form, one
// write per row, no atomics; Sec. 3.5 apply, Sec. 5.2 two-table index) as
// device functions, shared by k_apply (xd_u1.cu) and the persistent Lanczos
// kernel (xd_lanczos.cu).  For row r with state s and every bond b: equal
// spins add +J_b/4 x_r, opposite spins -J_b/4 x_r and +J_b/2 x_c with
// c = index(s ^ m_b); the diagonal is J_sum/4 - sum over flipped bonds J_b/2.

#pragma once

#include "xd_internal.cuh"

namespace xd {

// a product and a fused multiply-add with their roundings fixed (no
// contraction left to the compiler), for arithmetic that two kernels must
// reproduce bit for bit
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }

namespace u1rows {

// largest h in [lo, hi] with hi_off[h] <= r (hi_off is non-decreasing)
__device__ __forceinline__ uint64_t find_block(const int64_t *__restrict__ hi_off, uint64_t lo,
                                               uint64_t hi, int64_t r) {
    while (lo < hi) {
        uint64_t mid = (lo + hi + 1) >> 1;
        if (__ldg(hi_off + mid) <= r) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// The same by a warp, 32 entries at a time: a search of 2^P entries costs
// P / 5 dependent reads and not P.
__device__ __forceinline__ uint64_t find_block_warp(const int64_t *__restrict__ hi_off, uint64_t lo, uint64_t hi, int64_t r) {
    const uint64_t lane = threadIdx.x & 31;
    while (lo < hi) {
        const uint64_t step = (hi - lo + 32) / 32, at = lo + (lane + 1) * step;
        const uint32_t below = __ballot_sync(0xffffffffu, at <= hi && __ldg(hi_off + (at <= hi ? at : hi)) <= r);
        lo += __popc(below) * step;
        hi = min(hi, lo + step - 1);
    }
    return lo;
}

// Row r -> (state, block).  The CTA first brackets the blocks of its rows, its
// first two warps an end each (product of the 16-site chain, 51 CTAs: 9.4 ->
// 8.2 us).
struct RowState {
    uint64_t s;
    bool valid;
};

__device__ __forceinline__ RowState unrank_tile(const U1View &u, int64_t base, int64_t r,
                                                uint64_t *sh_range) {
    // sh_range[0..1]: block range of rows [base, base + blockDim.x)
    __syncthreads();
    if (threadIdx.x < 64) {
        const int64_t last = min(base + (int64_t)blockDim.x, u.dim) - 1;
        const uint64_t h = find_block_warp(u.hi_off, 0, (1ull << u.P) - 1, threadIdx.x < 32 ? base : last);
        if ((threadIdx.x & 31) == 0) sh_range[threadIdx.x >> 5] = h;
    }
    __syncthreads();
    RowState rs;
    rs.valid = r < u.dim;
    rs.s = 0;
    if (rs.valid) {
        uint64_t h = find_block(u.hi_off, sh_range[0], sh_range[1], r);
        int64_t i = r - __ldg(u.hi_off + h);
        int m = u.nup - __popcll(h);
        uint32_t l = __ldg(u.lo_list + __ldg(u.lo_off + m) + (uint32_t)i);
        rs.s = (h << u.L) | l;
    }
    return rs;
}

__device__ __forceinline__ int64_t rank_of(const U1View &u, uint64_t t) {
    return __ldg(u.hi_off + (t >> u.L)) + (int64_t)__ldg(u.lo_rank + (t & u.lomask));
}

// x entries: through the read-only path, or (COHERENT) through L2, for a
// vector written earlier by other CTAs of the same kernel; VEC: the vectors are
// 16-byte aligned and a row of NV entries is read and written in 16-byte pieces.
template <typename T, int NV>
constexpr bool kVecRow = (NV * sizeof(T)) % 16 == 0;

template <typename T, int NV, bool COHERENT, bool VEC>
__device__ __forceinline__ void load_row(const T *x, int64_t c, T (&out)[NV]) {
    if constexpr (VEC && kVecRow<T, NV>) {
        constexpr int P = 16 / (int)sizeof(T);
        const int4 *p = (const int4 *)(x + c * NV);
#pragma unroll
        for (int k = 0; k < NV / P; ++k) {
            const int4 q = COHERENT ? __ldcg(p + k) : __ldg(p + k);
            const T *v = (const T *)&q;
#pragma unroll
            for (int i = 0; i < P; ++i) out[k * P + i] = v[i];
        }
    } else {
#pragma unroll
        for (int k = 0; k < NV; ++k) out[k] = COHERENT ? __ldcg(x + c * NV + k) : __ldg(x + c * NV + k);
    }
}

template <typename T, int NV, bool VEC>
__device__ __forceinline__ void store_row(T *y, int64_t r, const T (&v)[NV]) {
    if constexpr (VEC && kVecRow<T, NV>) {
        constexpr int P = 16 / (int)sizeof(T);
#pragma unroll
        for (int k = 0; k < NV / P; ++k) {
            union {
                int4 q;
                T t[P];
            } w;
#pragma unroll
            for (int i = 0; i < P; ++i) w.t[i] = v[k * P + i];
            ((int4 *)(y + r * NV))[k] = w.q;
        }
    } else {
#pragma unroll
        for (int k = 0; k < NV; ++k) y[r * NV + k] = v[k];
    }
}

// A bond's J/2; FP32 also has it in units of 2^-30 of a power of two above sum
// |J/2|, for the diagonal.
template <typename T>
struct BondCoef {
    T h;
};
template <>
struct __align__(8) BondCoef<float> {
    float h;
    int f;
};

// The diagonal of a row, sum J/4 - sum over its flipping bonds of J/2.  The two
// sums cancel to a few J, so FP32 takes them in the integers above: an integer
// addition costs what an FP32 one does, and the error against 64 bits of a product
// with random couplings falls (23 sites, 103 bonds 5.2e-7 with FP32 sums).
template <typename T>
struct RowDiag {
    T jq;
    __device__ __forceinline__ RowDiag(const double *__restrict__ bond, int nb) : jq(bond[2 * nb]) {}
};
template <>
struct RowDiag<float> {
    const int4 *at;  // sum J/4 and the unit in two factors, both normal numbers: read for each row, registers being short
    __device__ __forceinline__ RowDiag(const double *__restrict__ bond, int nb) : at((const int4 *)(bond + (3 * nb + 3) / 2 * 2)) {}
};
template <typename T>
struct DiagSum {
    T s = T(0);
    __device__ __forceinline__ void add(BondCoef<T> c) { s += c.h; }
    __device__ __forceinline__ T diagonal(const RowDiag<T> &g) const { return g.jq - s; }
};
template <>
struct DiagSum<float> {
    int s = 0;
    __device__ __forceinline__ void add(BondCoef<float> c) { s += c.f; }
    __device__ __forceinline__ float diagonal(const RowDiag<float> &g) const {
        const int4 v = __ldg(g.at);
        return (float)(v.x - s) * __int_as_float(v.y) * __int_as_float(v.z);
    }
};

// The flipping bonds of a row with state s, in ascending order: acc += J_b/2
// x_c for each of the NV columns; d: the row's diagonal.  FP64 rows and rows of 32
// bytes and more (WALK): the bonds are tested 32 at a time and then only the
// set bits are walked, two targets being read together, so that a warp runs as
// long as its row with the most flips and not once for every bond with half of
// its lanes idle; the FP64 pipe, the limit in FP64, costs a warp the same
// whether lanes are idle or not.  fix (or null; [nb], and then the unit): J_b/2
// in integers, so that the diagonal costs that pipe one product a row and not one
// addition a flip.  FP64, in turn and now (us): 4x5 lattice, one column 55 and
// 33, two 76 and 50; 22-site ladder, one 104 and 69; 4x6 lattice, two 1066 and
// 706, eight 3058 and 2356 (2612 without the integers).  FP32, 22-site ladder,
// eight columns 175 -> 105.  One target at a time or four cost more (4x6
// lattice, eight 2586; 4x5, two 61).  Narrower FP32 rows take every bond in
// turn: the test is most of their work (22-site ladder, two FP32 columns: 52 us
// in turn, 66 us walked), and the integers cost them more than they save
// (FP64 in turn with them: 4x5 lattice 57 against 55).
template <typename T, int NV>
constexpr bool kWalkRow = sizeof(T) == 8 || NV * sizeof(T) >= 32;

template <typename T, int NV, bool COHERENT, bool VEC, bool WALK = kWalkRow<T, NV>>
__device__ __forceinline__ void row_flips(const U1View &u, uint64_t s, const uint64_t *sm_mask, const BondCoef<T> *sm_coef,
                                          int nb, const T *x, T (&acc)[NV], const RowDiag<T> &diag, T &d,
                                          const long long *fix = nullptr) {
    constexpr int D = 2;
    long long sum = 0;
    DiagSum<T> dsub;
    if constexpr (!WALK) {
        for (int b = 0; b < nb; ++b) {
            const uint64_t mk = sm_mask[b], t = s & mk;
            if (t != 0 && t != mk) {
                const BondCoef<T> c = sm_coef[b];
                T xv[NV];
                load_row<T, NV, COHERENT, VEC>(x, rank_of(u, s ^ mk), xv);
#pragma unroll
                for (int k = 0; k < NV; ++k) acc[k] = fma_rn(c.h, xv[k], acc[k]);
                dsub.add(c);
            }
        }
    } else {
        for (int b0 = 0; b0 < nb; b0 += 32) {
            uint32_t fl = 0;
            const int bn = min(32, nb - b0);
            for (int b = 0; b < bn; ++b) {
                const uint64_t mk = sm_mask[b0 + b], t = s & mk;
                fl |= (uint32_t)(t != 0 && t != mk) << b;
            }
            while (fl) {
                bool on[D];
                T cf[D], xv[D][NV];
#pragma unroll
                for (int d = 0; d < D; ++d) {
                    on[d] = fl != 0;
                    if (on[d]) {
                        const int b = b0 + __ffs(fl) - 1;
                        fl &= fl - 1;
                        const BondCoef<T> c = sm_coef[b];
                        cf[d] = c.h;
                        if constexpr (sizeof(T) == 4) dsub.add(c);
                        if (fix) sum += fix[b];
                        load_row<T, NV, COHERENT, VEC>(x, rank_of(u, s ^ sm_mask[b]), xv[d]);
                    }
                }
#pragma unroll
                for (int d = 0; d < D; ++d)
                    if (on[d]) {
#pragma unroll
                        for (int k = 0; k < NV; ++k) acc[k] = fma_rn(cf[d], xv[d][k], acc[k]);
                        if constexpr (sizeof(T) == 8) {
                            if (!fix) dsub.s += cf[d];
                        }
                    }
            }
        }
    }
    if constexpr (WALK && sizeof(T) == 8) {
        if (fix) dsub.s = (double)sum * __longlong_as_double(fix[nb]);
    }
    d = dsub.diagonal(diag);
}

// FP64 rows take the integer J_b/2 in shared memory, up to this many bonds and
// where the couplings have a unit.
constexpr int kFixBonds = 2048;
template <typename T>
constexpr bool kFixRow = sizeof(T) == 8;

// Bond masks and J_b/2 from the handle's bond table [J (nb) | masks (nb) | sum
// J / 4 | unit | J/2 in units (nb) | at the next multiple of 16 bytes, FP32: sum J / 4
// in units 2^32 times as large, that unit's two factors]; sm_fix: [nb + 1], or null.
template <typename T>
__device__ __forceinline__ void stage_bonds(const double *__restrict__ bond, int nb, uint64_t *sm_mask, BondCoef<T> *sm_coef,
                                            long long *sm_fix = nullptr) {
    const uint64_t *masks = (const uint64_t *)(bond + nb);
    if (sm_fix)
        for (int b = threadIdx.x; b <= nb; b += blockDim.x)
            sm_fix[b] = __double_as_longlong(b < nb ? bond[2 * nb + 2 + b] : bond[2 * nb + 1]);
    for (int b = threadIdx.x; b < nb; b += blockDim.x) {
        sm_coef[b].h = (T)(0.5 * bond[b]);
        if constexpr (sizeof(T) == 4) sm_coef[b].f = (int)((__double_as_longlong(bond[2 * nb + 2 + b]) + (1ll << 31)) >> 32);
        sm_mask[b] = masks[b];
    }
}

// y = H x on the rows of this CTA (grid-stride tiles of blockDim.x rows);
// every thread of the CTA calls it (the tile unranking has barriers).
template <typename T, int NV, bool COHERENT, bool VEC>
__device__ __forceinline__ void apply_rows(const U1View &u, const uint64_t *sm_mask, const BondCoef<T> *sm_coef, int nb,
                                           const RowDiag<T> &diag, const T *x, T *y, uint64_t *sh_range, const long long *fix) {
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < u.dim; base += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = base + threadIdx.x;
        const RowState rs = unrank_tile(u, base, r, sh_range);
        if (!rs.valid) continue;
        const uint64_t s = rs.s;
        T acc[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) acc[k] = T(0);
        T d;
        row_flips<T, NV, COHERENT, VEC>(u, s, sm_mask, sm_coef, nb, x, acc, diag, d, fix);
        T xr[NV];
        load_row<T, NV, COHERENT, VEC>(x, r, xr);
#pragma unroll
        for (int k = 0; k < NV; ++k) xr[k] = fma_rn(d, xr[k], acc[k]);
        store_row<T, NV, VEC>(y, r, xr);
    }
}

}  // namespace u1rows
}  // namespace xd
