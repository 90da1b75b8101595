// xd_u1.cu -- y = H x and per-bond bilinear forms on U(1) blocks.
//
// Pull form (the "apply" of Sec. 3.5 with the vector fill of Sec. 5.1):
// every row r of y is written once, no atomics.  For row r with state s
// (a1: unranked from the two-table layout, Sec. 5.2) and every bond b:
//   a2  equal spins:     +J_b/4 x_r on the diagonal
//   a3  opposite spins:  -J_b/4 x_r and +J_b/2 x_c, c = index(s ^ m_b)
//   a4  c from the prefix/postfix tables: c = hi_off[s'>>L] + lo_rank[s'&mask]
//   a5  gather x_c and accumulate.
// The diagonal is written as J_sum/4 - sum over flipped bonds of J_b/2.

#include <algorithm>
#include <mutex>

#include "xd_internal.cuh"
#include "xd_u1_rows.cuh"

namespace xd {

namespace {

constexpr int kThreads = 256;

using namespace u1rows;

// y = H x (the row loop of xd_u1_rows.cuh).  Eight FP32 columns in 48 registers,
// five CTAs to an SM (us, in 60: 20 sites with 100 bonds 80 and 97, 21 sites 134 and
// 144, 23 sites 506 and 445).
template <typename T, int NV, bool VEC>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 4 && NV == 8 ? 5 : 0) k_apply(U1View u, const double *__restrict__ bond,
                                                    int nb, const T *__restrict__ x,
                                                    T *__restrict__ y) {
    extern __shared__ __align__(16) unsigned char smem[];
    uint64_t *sm_mask = (uint64_t *)smem;
    BondCoef<T> *sm_coef = (BondCoef<T> *)(sm_mask + nb);
    __shared__ uint64_t sh_range[2];
    const bool fixed = kFixRow<T> && nb <= kFixBonds && bond[2 * nb + 1] != 0.0;
    long long *sm_fix = fixed ? (long long *)(sm_coef + nb) : nullptr;
    stage_bonds(bond, nb, sm_mask, sm_coef, sm_fix);
    const RowDiag<T> diag(bond, nb);
    __syncthreads();
    apply_rows<T, NV, false, VEC>(u, sm_mask, sm_coef, nb, diag, x, y, sh_range, sm_fix);
}

// State words of rows [first, first + count): the block of row r is the last
// h with hi_off[h] <= r (binary search), its word (h << L) | lo_list[...].
__global__ void k_states_range(U1View u, int64_t first, int64_t count, uint64_t *__restrict__ out) {
    const uint64_t nh = 1ull << u.P;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < count;
         q += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = first + q;
        const uint64_t h = find_block(u.hi_off, 0, nh - 1, r);
        const int m = u.nup - __popcll(h);
        const uint32_t l = __ldg(u.lo_list + __ldg(u.lo_off + m) + (uint32_t)(r - __ldg(u.hi_off + h)));
        out[q] = (h << u.L) | l;
    }
}

// Bonds per launch of the bilinear kernel, the most that a warp's share of
// them touches, rows per tile, CTAs per SM.
constexpr int kChunk = 64, kShare = 5, kBT = 512, kBPer = 4;

struct BilShared {
    uint64_t s[kBT], mask[kChunk];
    double g[kBT];
    long long p[kBT];  // fixed point, or the bits of the double
    uint16_t list[kBT / 32][kBT];
    double acc[kBT / 32][kShare][32];  // F_b - F'_b below, a lane's part
    double red[kBT / 32];
    uint32_t top[kBT / 32];
    uint64_t range[2];
};

// Per-bond bilinear forms: part[cta][b] = sum over the CTA's rows of
// g_r (S_i.S_j x)_r (Sec. 3.7 inner, per bond).  With p_r = g_r x_r and
// P = sum_r p_r,
//   <g|S_i.S_j|x> = 1/4 sum_r eps_b(s_r) p_r + 1/2 sum_{r: b flips} g_r x_c
//                 = 1/4 P + 1/2 (F_b - F'_b),
// F'_b = sum over flipping rows of p_r and F_b = sum over them of g_r x_c
// (eps = +1 for parallel, -1 for antiparallel spins): only the flipping
// bonds of a row cost arithmetic.  A CTA stages the states, g and p of a
// tile of kBT rows in shared memory; the bonds times the tile's 16 groups of
// 32 rows are dealt to the 16 warps in equal shares, a warp's share being up to
// kShare neighbouring bonds, the first and last of them in part.  All sums run in
// a fixed order (lane partials, a fixed shuffle tree, the warps of a bond, then
// the CTAs).
//
// The FP64 pipe (two lanes a clock and SM, idle lanes included) was the limit
// of one FP64 addition and one FMA for every row and bond with half of the
// lanes idle.  So a warp first lists the flipping rows of its bond and then
// takes 32 of them at a time, and F' is summed in integers: p is scaled by a
// power of two to 58 bits of the tile's largest |p|, whose sums over a lane's
// 16 rows are exact; the scaling loses less than an FP64 sum of them does.  A
// tile with an infinity, a NaN or only tiny p (below 2^-965) adds in FP64.
// The equal shares, sums kept in shared memory and 32 registers (64 warps on
// an SM) hide the look-ups; more look-ups in flight per lane cost more in idle
// lanes than they hide (two: 5.3 ms, four: 6.2 below), and a ring of 64 rows in
// place of the list 5.4.  28-site ladder, 56 bonds: FP64 8.25 -> 4.53 ms, FP32
// 11.2 -> 6.7 (the conversions); 4x7 lattice, 112 bonds, FP64 14.6 -> 9.1;
// diagonal part alone (ZZ), 28 pairs 3.7 -> 1.2.
template <typename T, bool ZZ>
__global__ void __launch_bounds__(kBT, kBPer)
    k_bilinear_bp(U1View u, const uint64_t *__restrict__ masks, int nb, int b0, const T *__restrict__ g,
                  const T *__restrict__ x, double *__restrict__ part, int nv) {
    // nv > 1: column of row-major [dim][nv] vectors (g, x point at the column)
    constexpr int kWarps = kBT / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    BilShared &sh = *(BilShared *)smem;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t below = (1u << lane) - 1;
    const int nbc = min(kChunk, nb - b0);
    const int share = warp * nbc, bf = share / kWarps;  // first group of this warp's share, and its bond
    uint16_t *const list = sh.list[warp];
    if (tid < nbc) sh.mask[tid] = __ldg(masks + b0 + tid);
    for (int j = 0; j < kShare; ++j) sh.acc[warp][j][lane] = 0.0;
    double P = 0.0;
    for (int64_t base = (int64_t)blockIdx.x * kBT; base < u.dim; base += (int64_t)gridDim.x * kBT) {
        const int64_t r = base + tid;
        const RowState rs = unrank_tile(u, base, r, sh.range);
        const double gr = rs.valid ? (double)g[r * nv] : 0.0;
        const double pr = rs.valid ? gr * (double)x[r * nv] : 0.0;
        P += pr;
        sh.s[tid] = rs.s;  // 0, a state without flips, beyond the last row
        sh.g[tid] = gr;
        const uint32_t wtop = __reduce_max_sync(0xffffffffu, (uint32_t)__double2hiint(fabs(pr)) >> 20);
        if (lane == 0) sh.top[warp] = wtop;
        __syncthreads();
        int top = 0;  // biased exponent of the largest |p|
#pragma unroll
        for (int w = 0; w < kWarps; ++w) top = max(top, (int)sh.top[w]);
        const bool fixed = top >= 58 && top < 2047;
        sh.p[tid] = fixed ? __double2ll_rn(pr * __hiloint2double((2103 - top) << 20, 0)) : __double_as_longlong(pr);
        const double unit = fixed ? __hiloint2double((top - 57) << 20, 0) : 0.0;
        __syncthreads();
        const int steps = (int)(min((int64_t)kBT, u.dim - base) + 31) / 32;
        for (int j = 0; j < kShare; ++j) {
            const int k0 = max(0, share - kWarps * (bf + j)), k1 = min(steps, share + nbc - kWarps * (bf + j));
            if (k0 >= k1) continue;
            const uint64_t mk = sh.mask[bf + j];
            double acc = sh.acc[warp][j][lane], direct = 0.0;
            long long sum = 0;
            int n = 0;
#pragma unroll 4
            for (int k = k0; k < k1; ++k) {
                const int rr = 32 * k + lane;
                const uint64_t t = sh.s[rr] & mk;
                const bool fl = t != 0 && t != mk;
                if (fl) sum += sh.p[rr];
                if (!ZZ) {
                    const uint32_t set = __ballot_sync(0xffffffffu, fl);
                    if (fl) list[n + __popc(set & below)] = (uint16_t)rr;
                    n += __popc(set);
                }
            }
            if (fixed) {
                acc = fma((double)sum, -unit, acc);
            } else {
#pragma unroll 1
                for (int k = k0; k < k1; ++k) {
                    const int rr = 32 * k + lane;
                    const uint64_t t = sh.s[rr] & mk;
                    if (t != 0 && t != mk) direct += __longlong_as_double(sh.p[rr]);
                }
                acc -= direct;
            }
            if (!ZZ) {
                __syncwarp();
                for (int i = lane; i < n; i += 32) {
                    const int rr = list[i];
                    acc = fma(sh.g[rr], (double)__ldg(x + rank_of(u, sh.s[rr] ^ mk) * nv), acc);
                }
                __syncwarp();
            }
            sh.acc[warp][j][lane] = acc;
        }
        // the next tile overwrites the staged rows after unrank_tile's barrier
    }
    for (int j = 0; j < kShare; ++j) {
        double v = sh.acc[warp][j][lane];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sh.acc[warp][j][0] = v;
    }
    for (int o = 16; o > 0; o >>= 1) P += __shfl_xor_sync(0xffffffffu, P, o);
    if (lane == 0) sh.red[warp] = P;
    __syncthreads();
    if (tid < nbc) {
        double Pb = 0.0, Fb = 0.0;
        for (int w = 0; w < kWarps; ++w) {
            Pb += sh.red[w];
            const int j = tid - w * nbc / kWarps;
            if (j >= 0 && kWarps * tid < (w + 1) * nbc) Fb += sh.acc[w][j][0];
        }
        part[(size_t)blockIdx.x * nb + b0 + tid] = 0.25 * Pb + 0.5 * Fb;
    }
}

// out[b] = sum_c part[c][b] in fixed order, a warp to a column.
__global__ void k_sum_columns(const double *__restrict__ part, int rows, int cols,
                              double *__restrict__ out) {
    const int b = (blockIdx.x * blockDim.x + threadIdx.x) / 32, lane = threadIdx.x & 31;
    if (b >= cols) return;
    double s = 0.0;
    for (int c = lane; c < rows; c += 32) s += part[(size_t)c * cols + b];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) out[b] = s;
}

}  // namespace

template <typename T, int NV>
static xd_status launch_apply(const xd_ham_s *h, const void *x, void *y, cudaStream_t st) {
    const double *bondbuf = h->d_bond;
    const U1View u = h->b->u1view();
    const int nb = h->b->nb;
    size_t smem = (size_t)nb * (sizeof(uint64_t) + sizeof(BondCoef<T>)) + (kFixRow<T> && nb <= kFixBonds ? (nb + 1) * sizeof(long long) : 0);
    auto kern = kVecRow<T, NV> && (((uintptr_t)x | (uintptr_t)y) & 15) == 0 ? k_apply<T, NV, kVecRow<T, NV>> : k_apply<T, NV, false>;
    if (smem > 48 * 1024) XD_CUDA(allow_smem(kern));
    int grid = grid_for(u.dim, kThreads, 8);
    kern<<<grid, kThreads, smem, st>>>(u, bondbuf, nb, (const T *)x, (T *)y);
    XD_CUDA(cudaGetLastError());
    return XD_OK;
}

xd_status u1_states(const xd_basis_s *b, int64_t first, int64_t count, uint64_t *out, cudaStream_t st) {
    const int grid = grid_for(count, kThreads, 8);
    k_states_range<<<grid, kThreads, 0, st>>>(b->u1view(), first, count, out);
    XD_CUDA(cudaGetLastError());
    return XD_OK;
}

xd_status u1_apply(const xd_ham_s *h, const void *x, void *y, xd_dtype dt, int nvec,
                   cudaStream_t st) {
    // window tables that do not fit in shared memory (very dense graphs) leave the
    // products to the kernels below, before anything is launched
    if (nvec == 1 && dt == XD_F32 && h->b->spmm.ok && (h->b->win.spmm32 || !h->win_fit[kWinF32])) return spmm_apply(h, x, y, st);
    if (nvec == 1 && dt == XD_F32 && h->win_fit[kWinF32]) return win_apply_f32(h, x, y, st);
    if (nvec == 1 && dt == XD_F64 && h->b->win.ok) {
        xd_status s = passes_wanted(h->b) ? passes_apply_f64(h, x, y, st) : XD_ERANGE;
        if (s == XD_ERANGE && h->win_fit[kWinF64]) s = win_apply_f64(h, x, y, st);
        // a workspace that does not fit sends this product to the block kernel
        if (s != XD_ENOMEM && s != XD_ERANGE) return s;
    }
    if (nvec == 8 && dt == XD_F32 && win8_usable(h, x, y)) return win8_apply(h, x, y, st);
    if (nvec == 8 && dt == XD_F32 && spmm8_usable(h, x, y)) return spmm8_apply(h, x, y, st);
    // (built below 24 sites for FP32 alone)
    if (nvec == 1 && h->b->blk.ok && (dt == XD_F32 || h->b->N >= 24)) return block_apply(h, x, y, dt, st);
    if (dt == XD_F64) {
        switch (nvec) {
            case 1: return launch_apply<double, 1>(h, x, y, st);
            case 2: return launch_apply<double, 2>(h, x, y, st);
            case 4: return launch_apply<double, 4>(h, x, y, st);
            default: return launch_apply<double, 8>(h, x, y, st);
        }
    }
    switch (nvec) {
        case 1: return launch_apply<float, 1>(h, x, y, st);
        case 2: return launch_apply<float, 2>(h, x, y, st);
        case 4: return launch_apply<float, 4>(h, x, y, st);
        default: return launch_apply<float, 8>(h, x, y, st);
    }
}

template <typename T, bool ZZ = false>
static xd_status launch_bilinear_bp(const U1View &u, const uint64_t *masks, int nb, int grid, const void *g,
                                    const void *x, double *part, cudaStream_t st, int nv = 1) {
    XD_CUDA(cudaFuncSetAttribute(k_bilinear_bp<T, ZZ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(BilShared)));
    for (int b0 = 0; b0 < nb; b0 += kChunk) {
        k_bilinear_bp<T, ZZ><<<grid, kBT, sizeof(BilShared), st>>>(u, masks, nb, b0, (const T *)g, (const T *)x, part, nv);
        XD_CUDA(cudaGetLastError());
    }
    return XD_OK;
}

// dJ[b] = sum over the nv columns of the per-bond forms: the partials of
// column k fill rows [k grid, (k + 1) grid) and one fixed-order sum over all
// rows follows (deterministic).
xd_status u1_bilinear_nvec(const xd_ham_s *h, const void *g, const void *x, xd_dtype dt, int nv, double *dJ,
                           cudaStream_t st) {
    const xd_basis_s *b = h->b;
    const int nb = b->nb;
    const U1View u = b->u1view();
    const int grid = grid_for(u.dim, kBT, kBPer);
    xd_ham_s *hm = const_cast<xd_ham_s *>(h);
    XD_TRY(ensure_partials(hm, sizeof(double) * (size_t)grid * nb * nv));
    const uint64_t *d_masks = (const uint64_t *)(h->d_bond + nb);
    const size_t es = dt == XD_F64 ? sizeof(double) : sizeof(float);
    for (int k = 0; k < nv; ++k) {
        const void *gk = (const char *)g + k * es, *xk = (const char *)x + k * es;
        double *pk = hm->d_part + (size_t)k * grid * nb;
        if (dt == XD_F64) XD_TRY(launch_bilinear_bp<double>(u, d_masks, nb, grid, gk, xk, pk, st, nv));
        else XD_TRY(launch_bilinear_bp<float>(u, d_masks, nb, grid, gk, xk, pk, st, nv));
    }
    k_sum_columns<<<(nb + 3) / 4, 128, 0, st>>>(hm->d_part, grid * nv, nb, dJ);
    XD_CUDA(cudaGetLastError());
    return XD_OK;
}

xd_status u1_bilinear(const xd_ham_s *h, const void *g, const void *x, xd_dtype dt, double *dJ,
                      cudaStream_t st) {
    const xd_basis_s *b = h->b;
    const int nb = b->nb;
    const U1View u = b->u1view();
    const int grid = grid_for(u.dim, kBT, kBPer);
    xd_ham_s *hm = const_cast<xd_ham_s *>(h);
    XD_TRY(ensure_partials(hm, sizeof(double) * (size_t)grid * nb));
    const uint64_t *d_masks = (const uint64_t *)(h->d_bond + nb);
    double *d_part = hm->d_part;
    if (dt == XD_F64) XD_TRY(launch_bilinear_bp<double>(u, d_masks, nb, grid, g, x, d_part, st));
    else XD_TRY(launch_bilinear_bp<float>(u, d_masks, nb, grid, g, x, d_part, st));
    k_sum_columns<<<(nb + 3) / 4, 128, 0, st>>>(d_part, grid, nb, dJ);
    XD_CUDA(cudaGetLastError());
    return XD_OK;
}


// ---------------------------------------------------------------------------
// Allocation-free variant of the per-bond bilinear forms.
//
// Some callers cannot let a library call cudaMalloc: a process whose own
// allocator owns all device memory (a pool sized once at start-up, or a hard
// memory budget), or a latency-sensitive loop where cudaMalloc/cudaFree may
// synchronise the device.  xd_apply_bilinear keeps its per-CTA partial sums
// in a workspace that the handle allocates (and grows) on demand; this
// variant keeps them in the fixed file-scope array below instead, so the
// call itself allocates nothing.  Every call, on every stream, shares this
// one array and leaves the last call's partials in it; nothing in it needs
// to start at zero (each launch writes every partial it later reads), but
// two calls that overlap on the GPU race on it and give wrong results.

namespace {

// [kNoAllocCtas][kNoAllocBonds] partial sums: 608 x 256 doubles = 1.19 MiB,
// held on every GPU that loads the library until the process exits.
constexpr int kNoAllocCtas = 608;
constexpr int kNoAllocBonds = 256;
static __device__ __align__(256) double g_noalloc_partials[kNoAllocCtas * kNoAllocBonds];

constexpr int kMaxDevices = 64;
std::mutex g_noalloc_mu;
double *g_noalloc_ptr[kMaxDevices] = {};

// Device address of the array on the current device.  In host code the name
// g_noalloc_partials is only a host-side stand-in, so the address comes from
// cudaGetSymbolAddress, once per device, with that device current.
xd_status noalloc_scratch(double **out) {
    int dev = 0;
    XD_CUDA(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMaxDevices) {
        set_error("xd_apply_bilinear_noalloc: device %d beyond the %d supported", dev, kMaxDevices);
        return XD_ERANGE;
    }
    std::lock_guard<std::mutex> lk(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
        void *p = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_partials);
        if (e != cudaSuccess) return cuda_status(e, "cudaGetSymbolAddress(g_noalloc_partials)");
        g_noalloc_ptr[dev] = (double *)p;
    }
    *out = g_noalloc_ptr[dev];
    return XD_OK;
}

}  // namespace

}  // namespace xd

extern "C" xd_status xd_apply_bilinear_noalloc(xd_ham h, const void *g, const void *x, xd_dtype dt,
                                               double *dJ, xd_stream stream) {
    using namespace xd;
    if (!h || !g || !x || !dJ) {
        set_error("xd_apply_bilinear_noalloc: NULL argument");
        return XD_EINVAL;
    }
    const xd_basis_s *b = h->b;
    if (b->sym) {
        set_error("xd_apply_bilinear_noalloc: U(1) blocks only (this block is symmetry-adapted)");
        return XD_EINVAL;
    }
    if (dt != XD_F64 && dt != XD_F32) {
        set_error("xd_apply_bilinear_noalloc: dtype must be XD_F64 or XD_F32");
        return XD_EINVAL;
    }
    const int nb = b->nb;
    if (nb > kNoAllocBonds) {
        set_error("xd_apply_bilinear_noalloc: %d bonds exceed the fixed scratch limit of %d bonds "
                  "(use xd_apply_bilinear)", nb, kNoAllocBonds);
        return XD_ERANGE;
    }
    if (b->dim == 0) return XD_OK;
    double *part = nullptr;
    XD_TRY(noalloc_scratch(&part));
    const U1View u = b->u1view();
    const int grid = std::min(grid_for(u.dim, kBT, kBPer), kNoAllocCtas);
    const uint64_t *masks = (const uint64_t *)(h->d_bond + nb);
    cudaStream_t st = (cudaStream_t)stream;
    if (dt == XD_F64) XD_TRY(launch_bilinear_bp<double>(u, masks, nb, grid, g, x, part, st));
    else XD_TRY(launch_bilinear_bp<float>(u, masks, nb, grid, g, x, part, st));
    k_sum_columns<<<(nb + 3) / 4, 128, 0, st>>>(part, grid, nb, dJ);
    XD_CUDA(cudaGetLastError());
    return XD_OK;
}

// Two-point spin correlations out[p] = <psi| O_{i_p j_p} |psi> on a U(1)
// block: the bilinear kernel with g = x = psi and the pair masks as bonds
// (S_i.S_j), or its diagonal part alone (Sz_i Sz_j, no gathers).  A pair
// with i = j has a one-bit mask that never flips: the kernel returns
// <psi|psi>/4, which is (Sz_i)^2; S_i.S_i = 3/4 is three times that.
extern "C" xd_status xd_correlations(xd_basis b, const void *psi, xd_dtype dt, const int32_t *pairs,
                                     int npairs, int kind, double *out) {
    using namespace xd;
    if (!b || !psi || !out || (npairs > 0 && !pairs)) {
        set_error("xd_correlations: NULL argument");
        return XD_EINVAL;
    }
    if (b->sym ? dt != (b->cplx ? XD_C128 : XD_F64) : (dt != XD_F64 && dt != XD_F32)) {
        set_error(b->sym ? "xd_correlations: a symmetric block takes XD_F64 (real) or XD_C128 (complex)"
                         : "xd_correlations: dtype must be XD_F64 or XD_F32");
        return XD_EINVAL;
    }
    if (kind != 0 && kind != 1) {
        set_error("xd_correlations: kind must be 0 (Sz Sz) or 1 (S.S)");
        return XD_EINVAL;
    }
    if (npairs < 0 || npairs > (1 << 20)) {
        set_error("xd_correlations: npairs = %d out of range", npairs);
        return XD_ERANGE;
    }
    std::vector<uint64_t> m(npairs);
    for (int q = 0; q < npairs; ++q) {
        const int i = pairs[2 * q], j = pairs[2 * q + 1];
        if (i < 0 || i >= b->N || j < 0 || j >= b->N) {
            set_error("xd_correlations: pair %d = (%d, %d) outside 0..%d", q, i, j, b->N - 1);
            return XD_EINVAL;
        }
        m[q] = (1ull << i) | (1ull << j);
    }
    if (npairs == 0) return XD_OK;
    if (b->dim == 0) {
        for (int q = 0; q < npairs; ++q) out[q] = 0.0;
        return XD_OK;
    }
    if (b->sym) return sym_correlations(b, psi, dt, pairs, npairs, kind, out);
    const U1View u = b->u1view();
    const int grid = grid_for(u.dim, kBT, kBPer);
    uint64_t *d_m = nullptr;
    double *d_part = nullptr, *d_out = nullptr;
    cudaError_t e = dev_malloc((void **)&d_m, sizeof(uint64_t) * npairs);
    if (e == cudaSuccess) e = dev_malloc((void **)&d_part, sizeof(double) * (size_t)grid * npairs);
    if (e == cudaSuccess) e = dev_malloc((void **)&d_out, sizeof(double) * npairs);
    if (e == cudaSuccess) e = cudaMemcpy(d_m, m.data(), sizeof(uint64_t) * npairs, cudaMemcpyHostToDevice);
    xd_status s = e == cudaSuccess ? XD_OK : cuda_status(e, "xd_correlations workspace");
    if (s == XD_OK) {
        if (dt == XD_F64)
            s = kind ? launch_bilinear_bp<double, false>(u, d_m, npairs, grid, psi, psi, d_part, 0)
                     : launch_bilinear_bp<double, true>(u, d_m, npairs, grid, psi, psi, d_part, 0);
        else
            s = kind ? launch_bilinear_bp<float, false>(u, d_m, npairs, grid, psi, psi, d_part, 0)
                     : launch_bilinear_bp<float, true>(u, d_m, npairs, grid, psi, psi, d_part, 0);
    }
    if (s == XD_OK) {
        k_sum_columns<<<(npairs + 3) / 4, 128>>>(d_part, grid, npairs, d_out);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpy(out, d_out, sizeof(double) * npairs, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) s = cuda_status(e, "xd_correlations");
    }
    cudaFree(d_m);
    cudaFree(d_part);
    cudaFree(d_out);
    if (s != XD_OK) return s;
    if (kind)
        for (int q = 0; q < npairs; ++q)
            if (pairs[2 * q] == pairs[2 * q + 1]) out[q] *= 3.0;
    return XD_OK;
}

namespace xd {
}  // namespace xd
