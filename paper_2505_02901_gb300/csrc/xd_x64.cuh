// xd_x64.cuh -- FP64 products without FP64 arithmetic per matrix element:
// double-float pieces, the statistics of x, the choice of arithmetic and the
// conversion, and the quantum of the couplings (xd_u1_win.cu describes the
// two arithmetics; xd_u1_passes.cu uses them too).
#pragma once

#include <algorithm>
#include <numeric>
#include <vector>

#include "xd_internal.cuh"

namespace xd {

namespace {

constexpr int kStatThreads = 256;
constexpr int kStatPerSm = 8;

// ------------------------------------------------------ double-float pieces
// (s, c) += (C + gamma) (hi + lo): exact product of the leading parts,
// TwoSum into s, every rounding error and the small terms into c.
__device__ __forceinline__ void df_fma(float &s, float &c, float2 C, float2 v) {
    const float p = __fmul_rn(C.x, v.x);
    const float e = __fmaf_rn(C.x, v.x, -p);
    const float low = __fmaf_rn(C.y, v.x, __fmaf_rn(C.x, v.y, e));
    const float t = __fadd_rn(s, p);
    const float bp = __fsub_rn(t, s);
    const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(p, bp));
    s = t;
    c = __fadd_rn(c, __fadd_rn(err, low));
}

__device__ __forceinline__ float2 df_add(float2 a, float2 b) {
    const float t = __fadd_rn(a.x, b.x);
    const float bp = __fsub_rn(t, a.x);
    const float err = __fadd_rn(__fsub_rn(a.x, __fsub_rn(t, bp)), __fsub_rn(b.x, bp));
    return make_float2(t, __fadd_rn(err, __fadd_rn(a.y, b.y)));
}

// the double 2^(E - 1023) f, built from the bits of f (exact; subnormal f
// is taken as zero); E must keep the result in the normal double range
__device__ __forceinline__ double f2d_scaled(float f, int E) {
    const uint32_t u = __float_as_uint(f);
    const int fe = (int)((u >> 23) & 0xffu);
    const uint64_t sign = (uint64_t)(u >> 31) << 63;
    if (fe == 0) return __longlong_as_double((long long)sign);
    return __longlong_as_double((long long)(sign | ((uint64_t)(fe - 127 + E) << 52) | ((uint64_t)(u & 0x7fffffu) << 29)));
}

// 2^(E - 1023) (s + c).  For 300 <= E <= 1700 both words fold the scale into
// their exponents exactly (every float exponent stays inside the normal
// double range) and one FP64 addition rounds the sum.  Otherwise (vectors
// near the ends of the double range) the unscaled sum is multiplied by
// 2^(E - 1023) in FP64, which rounds correctly into the subnormal range or
// to infinity.  E = 2047 (x not finite) gives NaN.
__device__ __forceinline__ double df_result(float s, float c, int E) {
    if (E >= 300 && E <= 1700) return f2d_scaled(s, E) + f2d_scaled(c, E);
    if (E == 2047) return __longlong_as_double(0x7ff8000000000000ll);
    const double v = f2d_scaled(s, 1023) + f2d_scaled(c, 1023);
    return v * __longlong_as_double((long long)((uint64_t)E << 52));
}

// 2^k as a double for any k (two factors when 2^k is outside the normal range)
__device__ __forceinline__ double pow2d(int k, double v) {
    if (k >= -1022 && k <= 1023) return v * __longlong_as_double((long long)((uint64_t)(k + 1023) << 52));
    const int h = k / 2;
    v *= __longlong_as_double((long long)((uint64_t)(h + 1023) << 52));
    return v * __longlong_as_double((long long)((uint64_t)(k - h + 1023) << 52));
}

// 4^d for d <= 0 in FP32 (0 below the normal range)
__device__ __forceinline__ float pow4f(int d) { return 2 * d >= -126 ? __uint_as_float((uint32_t)(127 + 2 * d) << 23) : 0.f; }

struct ExpSum {
    int m;    // largest biased exponent seen
    float s;  // sum over the entries seen of 4^(e - m), e their biased exponents
};

__device__ __forceinline__ ExpSum es_join(ExpSum a, ExpSum b) {
    if (a.m == 2047 || b.m == 2047) return ExpSum{2047, 0.f};
    const int m = max(a.m, b.m);
    return ExpSum{m, a.s * pow4f(a.m - m) + b.s * pow4f(b.m - m)};
}

__device__ ExpSum es_block_reduce(ExpSum v) {
    __shared__ ExpSum red[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        ExpSum w;
        w.m = __shfl_xor_sync(0xffffffffu, v.m, o);
        w.s = __shfl_xor_sync(0xffffffffu, v.s, o);
        v = es_join(v, w);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) red[warp] = v;
    __syncthreads();
    if (warp == 0) {
        v = lane < nw ? red[lane] : ExpSum{0, 0.f};
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            ExpSum w;
            w.m = __shfl_xor_sync(0xffffffffu, v.m, o);
            w.s = __shfl_xor_sync(0xffffffffu, v.s, o);
            v = es_join(v, w);
        }
        if (lane == 0) red[0] = v;
    }
    __syncthreads();
    return red[0];
}

// Per CTA: the largest biased exponent of its entries of x (2047 when one is
// infinite or NaN) and sum 4^(e - m) over them, which bounds |x|^2 from
// below within a factor of 4 (zero and subnormal entries count as zero).
__global__ void k_x64_stats(const unsigned long long *__restrict__ x, int64_t n, ExpSum *__restrict__ part) {
    ExpSum v{0, 0.f};
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const int e = (int)((__ldg(x + i) >> 52) & 0x7ffull);
        if (e == 0) continue;
        if (e == 2047) v.m = 2047;
        if (v.m == 2047) continue;
        if (e > v.m) {
            v.s = v.s * pow4f(v.m - e) + 1.f;
            v.m = e;
        } else {
            v.s += pow4f(e - v.m);
        }
    }
    v = es_block_reduce(v);
    if (threadIdx.x == 0) part[blockIdx.x] = v;
}

// Every CTA joins the partials into E (largest biased exponent) and S, and
// takes the same decision: fixed point when allowed (the couplings have a
// quantum) and when rounding x to the grid 2^-S of the fixed point, at most
// sqrt(dim) 2^(E - 1023 - B) in norm, stays below 2^-44 |x| with |x|^2 >=
// 4^(E - 1023) S, i.e. dim / S <= 4^(B - 44); else double-float.  CTA 0
// records E and the decision for the product kernels; then x is converted
// (fixed point: X = round(2^S x), S = B - E + 1022, |X| < 2^B; double-float:
// (hi, lo) of 2^(1023 - E) x, hi the top 24 significant bits, lo the next 29
// rounded to FP32).  Subnormal doubles become zero in both.
__global__ void k_x64_convert(const unsigned long long *__restrict__ x, int64_t n, const ExpSum *__restrict__ part,
                              int npart, int fx_allowed, int B, int *__restrict__ state, void *__restrict__ out) {
    ExpSum v{0, 0.f};
    for (int c = threadIdx.x; c < npart; c += blockDim.x) v = es_join(v, part[c]);
    v = es_block_reduce(v);
    const int E = v.m;
    const bool fx = fx_allowed && E != 2047 && E != 0 &&
                    (double)n <= (double)v.s * ldexp(1.0, 2 * (B - 44));
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        state[0] = E;
        state[1] = fx ? 1 : 0;
    }
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const unsigned long long b = __ldg(x + i);
        const int e = (int)((b >> 52) & 0x7ffull);
        if (fx) {
            long long w = 0;
            if (e != 0) {
                const unsigned long long M = (b & 0xfffffffffffffull) | (1ull << 52);
                const int sh = e - E + B - 53;  // 2^S x = M 2^sh, sh <= B - 53
                if (sh >= 0) w = (long long)(M << sh);
                else if (sh > -64) w = (long long)((M >> (-sh)) + ((M >> (-sh - 1)) & 1ull));
                if (b >> 63) w = -w;
            }
            ((long long *)out)[i] = w;
        } else {
            const uint32_t sign = (uint32_t)(b >> 32) & 0x80000000u;
            const int fe = e - E + 127;  // FP32 exponent field of the scaled value
            float hi = 0.f, lo = 0.f;
            if (e != 0 && e != 2047 && fe > 0) {
                hi = __uint_as_float(sign | ((uint32_t)fe << 23) | (uint32_t)((b >> 29) & 0x7fffffull));
                const uint32_t r = (uint32_t)(b & 0x1fffffffull);  // value r 2^(fe - 127 - 52)
                if (r != 0 && fe - 52 > 0)
                    lo = __uint_as_float(sign | __float_as_uint(__uint2float_rn(r) *
                                                                __uint_as_float((uint32_t)(fe - 52) << 23)));
            }
            ((float2 *)out)[i] = make_float2(hi, lo);
        }
    }
}

// Statistics of x, the choice of arithmetic (state) and x in it (workspace).
inline void x64_convert(const xd_ham_s *h, const void *x, int64_t dim, cudaStream_t st) {
    const int g1 = grid_for(dim, kStatThreads, kStatPerSm);
    ExpSum *part = (ExpSum *)((unsigned char *)h->d_x64_state + 16);
    k_x64_stats<<<g1, kStatThreads, 0, st>>>((const unsigned long long *)x, dim, part);
    k_x64_convert<<<g1, kStatThreads, 0, st>>>((const unsigned long long *)x, dim, part, g1, h->x64_fx_ok ? 1 : 0,
                                               h->x64_B, h->d_x64_state, h->d_x64_x);
}

// Couplings as small integer multiples of one quantum: J_b = k_b q.  With
// J_b = m_b 2^e_b (m_b odd), q = gcd(m) 2^(min e); accepted when every |k_b|
// <= 2^16 and sum |k_b| <= 1365 (so that B >= 47).
inline bool find_quantum(const std::vector<double> &J, double *q, std::vector<int> *k) {
    int64_t g = 0;
    int emin = 1 << 20;
    std::vector<std::pair<int64_t, int>> me;
    for (double v : J) {
        if (v == 0.0) {
            me.push_back({0, 0});
            continue;
        }
        int e = 0;
        const double f = frexp(v, &e);             // v = f 2^e, 0.5 <= |f| < 1
        int64_t mm = (int64_t)ldexp(f, 53);        // exact: 53-bit integer
        e -= 53;
        while ((mm & 1) == 0) {
            mm /= 2;
            ++e;
        }
        me.push_back({mm, e});
        g = std::gcd(g, mm < 0 ? -mm : mm);
        emin = std::min(emin, e);
    }
    k->assign(J.size(), 0);
    if (g == 0) {
        *q = 1.0;
        return true;
    }
    int64_t kabs = 0;
    for (size_t b = 0; b < J.size(); ++b) {
        if (me[b].first == 0) continue;
        const int sh = me[b].second - emin;
        const int64_t mq = me[b].first / g;
        if (sh > 16 || mq > 65536 || mq < -65536) return false;
        const int64_t kb = mq * ((int64_t)1 << sh);
        if (kb > 65536 || kb < -65536) return false;
        (*k)[b] = (int)kb;
        kabs += kb < 0 ? -kb : kb;
        if (kabs > 1365) return false;
    }
    *q = ldexp((double)g, emin);
    return true;
}

}  // namespace

}  // namespace xd
