// bq_split.cu -- the hopping term (Eq. 1 / Eq. 5) with its clover epilogues and
// the CG-fused steps for small lattices: the work of one output site spread over
// eight threads, so that a lattice of a few thousand sites reaches every SM.
//
// With one thread per site (bq_stencil.cuh) an 8^4 lattice is 16 blocks on 152
// SMs: the FP64 launches wait for the FP64 pipe of those 16 SMs (GB300 issues
// about two FP64 lanes per clock and SM) and the FP32 ones for eight hops of
// dependent loads in a row. Here a block of four warps owns 16 sites. Warp mu
// takes the two hops along direction mu; the lanes 0-15 and 16-31 of a warp take
// the two projected half spinors, which are independent through the colour
// product (both halves read the same link addresses: one broadcast load). Every
// load of a site is in flight at once. The four partial spinors meet in shared
// memory; then thread (w, part, site) owns the real or imaginary part of the
// components w, w + 4, w + 8 for the sum, the clover rows and the stores, so no
// arithmetic is repeated: against one thread per site only 72 additions (the sums
// over the four warps) come on top of 1128 operations. FP64 Mhat^dag Mhat at 8^4:
// 158 us with one thread per site, 86 with two, 34 with eight; FP32 15.4 -> 13.4 us.
// Both hops' loads are issued before either's arithmetic (two resident blocks per SM are
// enough here; with the second hop's loads after the first's arithmetic 36 and 14.1 us;
// the clover rows' loads before the hops as well: 36 us).
//
// What bounds the FP64 launches: an FP64 warp instruction holds its scheduler's FP64
// pipe for about 64 cycles, so a launch takes whole rounds of (instructions per thread)
// x 64 cycles over the 608 schedulers. At 8^4 the eight-thread kernel is one round of
// 141 instructions (4.7 us of the 9 us a launch takes; the rest is load and launch
// latency). Two threads per site (k_dslash_pair64, 16 sites per warp, blocks of one warp)
// halve the rounds' length on larger lattices against one thread per site: 16^3x32 has 3.4
// rounds of 38 us (rounded up to 4, 614 us for Mhat^dag Mhat) or 6.7 of 19 us (541 us);
// 20^3x40 1366 -> 1288 us. With one pipe round per launch below that, three variants of
// block size for one thread per site (128, 64, 32) measured the same.
#include "bq_reduce.cuh"
#include "bq_split.cuh"

namespace {

constexpr int SPLIT_SITES = 16;

// component c (spin * 3 + colour) of the stored spinor at h; FP16: without the site's scale
template <int PREC>
__device__ __forceinline__ cplx<typename Traits<PREC>::real> load_comp(const void *base, int c, int h, int Vh) {
    if constexpr (PREC == BQ_PREC_DOUBLE) {
        const double2 v = ldg<true>(static_cast<const double2 *>(base) + (size_t)c * Vh + h);
        return {v.x, v.y};
    } else if constexpr (PREC == BQ_PREC_SINGLE) {
        const float2 v = ldg<true>(static_cast<const float2 *>(base) + ((size_t)(c >> 1) * Vh + h) * 2 + (c & 1));
        return {v.x, v.y};
    } else {
        const float2 v = h2f(ldg<true>(static_cast<const uint32_t *>(base) + ((size_t)(c >> 2) * Vh + h) * 4 + (c & 3)));
        return {v.x, v.y};
    }
}
template <int PREC>
__device__ __forceinline__ typename Traits<PREC>::real load_scale(const void *base, int h, int Vh) {
    if constexpr (PREC == BQ_PREC_HALF)
        return ldg<true>(reinterpret_cast<const float *>(static_cast<const uint4 *>(base) + (size_t)3 * Vh) + h);
    else
        return 1;
}
// address of real part (part 0) or imaginary part (1) of component c in FP32 / FP64 storage
template <typename T>
__device__ __forceinline__ size_t real_at(int c, int part, int h, int Vh) {
    return sizeof(T) == 8 ? ((size_t)c * Vh + h) * 2 + part : ((size_t)(c >> 1) * Vh + h) * 4 + 2 * (c & 1) + part;
}

// row i (0..11) of the clover term at h: the diagonal entry and the five others of its
// chirality block, B[i][j] for j != i in the order of j
template <int PREC>
struct CloverRow {
    using T = typename Traits<PREC>::real;
    T d;
    cplx<T> o[5];
    __device__ __forceinline__ void load(const void *base, int i, int h, int Vh) {
        const int b = i >= 6, ib = b ? i - 6 : i;
        if constexpr (PREC == BQ_PREC_DOUBLE)
            d = ldg(static_cast<const double *>(base) + ((size_t)(18 * b + (ib >> 1)) * Vh + h) * 2 + (ib & 1));
        else if constexpr (PREC == BQ_PREC_SINGLE)
            d = ldg(static_cast<const float *>(base) + ((size_t)(9 * b + (ib >> 2)) * Vh + h) * 4 + (ib & 3));
        else
            d = __half2float(__ushort_as_half(ldg(static_cast<const unsigned short *>(base) +
                                                  ((size_t)(9 * b + (ib >> 2)) * Vh + h) * 4 + (ib & 3))));
#pragma unroll
        for (int n = 0; n < 5; n++) {
            const int j = n + (n >= ib), r = ib < j ? ib : j, s = ib < j ? j : ib;
            const int e = r * (11 - r) / 2 + s - r - 1;  // packed upper entry (r, s)
            cplx<T> v;
            if constexpr (PREC == BQ_PREC_DOUBLE) {
                const double2 u = ldg(static_cast<const double2 *>(base) + (size_t)(18 * b + 3 + e) * Vh + h);
                v = {u.x, u.y};
            } else {
                const int k = 3 + e;  // entry as the k-th pair of reals of the block
                const size_t at = ((size_t)(9 * b + (k >> 1)) * Vh + h) * 2 + (k & 1);
                const float2 u = PREC == BQ_PREC_SINGLE ? ldg(static_cast<const float2 *>(base) + at)
                                                        : h2f(ldg(static_cast<const uint32_t *>(base) + at));
                v = {u.x, u.y};
            }
            o[n] = ib < j ? v : cconj(v);
        }
    }
    // the real (part 0) or imaginary (part 1) part of sum_j B[i][j] x_j; x: reals [24][SPLIT_SITES] at this site
    __device__ __forceinline__ T apply(const T *x, int i, int part) const {
        const int b = i >= 6, ib = b ? i - 6 : i;
        const T *xb = x + 12 * b * SPLIT_SITES;
        T y = d * xb[(2 * ib + part) * SPLIT_SITES];
#pragma unroll
        for (int n = 0; n < 5; n++) {
            const int j = n + (n >= ib);
            y = fma(o[n].re, xb[(2 * j + part) * SPLIT_SITES], y);
            y = fma(part ? o[n].im : -o[n].im, xb[(2 * j + 1 - part) * SPLIT_SITES], y);
        }
        return y;
    }
};

// One hop of half spinor q, its loads apart from its arithmetic so that a thread can have several
// hops' loads in flight. apply: up += f u, low += f times the lower spin that u feeds (FU, FL: set
// instead of added); f = the time-hop coefficient and the site's FP16 scale, one multiplier of the
// accumulating FMAs.
template <int PREC, int RECON, int MU, int S, bool BACK>
struct HalfHop {
    using T = typename Traits<PREC>::real;
    cplx<T> p[3], pj[3], U[9];
    T f;
    __device__ __forceinline__ void load(const void *in, int hn, const char *lblk, int hl, int Vh, int q, T coef) {
        const int jq = MU < 2 ? 3 - q : 2 + q;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            p[c] = load_comp<PREC>(in, 3 * q + c, hn, Vh);
            pj[c] = load_comp<PREC>(in, 3 * jq + c, hn, Vh);
        }
        f = MU == 3 ? coef : T(1);
        if (PREC == BQ_PREC_HALF) f *= load_scale<PREC>(in, hn, Vh);
        LinkIO<PREC, RECON>::load(U, lblk, hl, Vh);
    }
    template <bool FU, bool FL>
    __device__ __forceinline__ void apply(cplx<T> up[3], cplx<T> low[3], int q) const {
        constexpr bool SCALED = PREC == BQ_PREC_HALF || MU == 3;
        // the sign of the projector's off-diagonal factor differs between the halves for mu = y, z
        const T s = (MU == 0) ? T(-S) : (MU == 3) ? T(S) : (q ? T(S) : T(-S));
        cplx<T> h[3];
#pragma unroll
        for (int c = 0; c < 3; c++) {
            if (MU == 0 || MU == 2)  // p + i s pj
                h[c] = {fma(-s, pj[c].im, p[c].re), fma(s, pj[c].re, p[c].im)};
            else
                h[c] = {fma(s, pj[c].re, p[c].re), fma(s, pj[c].im, p[c].im)};
        }
        // the lower spin takes i S u (x), s u (y), -i s u (z), S u (t)
        const T g = (MU == 0) ? T(S) : (MU == 2) ? -s : s;
        const T gf = SCALED ? g * f : g;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            cplx<T> u = BACK ? cmulc(U[a], h[0]) : cmul(U[a * 3], h[0]);
#pragma unroll
            for (int b = 1; b < 3; b++) u = BACK ? cfmac(U[b * 3 + a], h[b], u) : cfma(U[a * 3 + b], h[b], u);
            const cplx<T> l = (MU == 0 || MU == 2) ? cplx<T>{-u.im, u.re} : u;
            if (FU) up[a] = SCALED ? cscale(f, u) : u;
            else up[a] = SCALED ? cplx<T>{fma(f, u.re, up[a].re), fma(f, u.im, up[a].im)} : cadd(up[a], u);
            if (FL) low[a] = cscale(gf, l);
            else low[a] = {fma(gf, l.re, low[a].re), fma(gf, l.im, low[a].im)};
        }
    }
};
template <int PREC, int RECON, int MU, int S, bool BACK, bool FU, bool FL>
__device__ __forceinline__ void half_hop(cplx<typename Traits<PREC>::real> up[3],
                                         cplx<typename Traits<PREC>::real> low[3], const void *in, int hn,
                                         const char *lblk, int hl, int Vh, int q,
                                         typename Traits<PREC>::real coef) {
    HalfHop<PREC, RECON, MU, S, BACK> x;
    x.load(in, hn, lblk, hl, Vh, q, coef);
    x.template apply<FU, FL>(up, low, q);
}

template <int PREC, int RECON, bool DAG, int MU>
__device__ __forceinline__ void two_hops(cplx<typename Traits<PREC>::real> up[3],
                                         cplx<typename Traits<PREC>::real> low[3], const DslashArgs &a, int h, int hf,
                                         int hb, int q, typename Traits<PREC>::real cf,
                                         typename Traits<PREC>::real cb) {
    constexpr int SF = DAG ? +1 : -1;
    const char *Lo = a.links + (size_t)a.parity * 4 * a.lblk + MU * a.lblk;
    const char *Li = a.links + (size_t)(1 - a.parity) * 4 * a.lblk + MU * a.lblk;
    HalfHop<PREC, RECON, MU, SF, false> fwd;
    HalfHop<PREC, RECON, MU, -SF, true> back;
    fwd.load(a.in, hf, Lo, h, a.Vh, q, cf);
    back.load(a.in, hb, Li, hb, a.Vh, q, cb);
    fwd.template apply<true, true>(up, low, q);
    back.template apply<false, false>(up, low, q);
}

// MODE 0, or the CG-fused steps of bq_cgfuse.cu (CNT_CG_MHAT / CNT_CG_MHATDAG, EPI_XPAY)
template <int PREC, int RECON, bool DAG, int EPI, int MODE>
__global__ void __launch_bounds__(128, 2) k_dslash_split(const DslashArgs a, const CgFuse f) {
    bq_pdl_enter();
    using T = typename Traits<PREC>::real;
    __shared__ T sp[4][24][SPLIT_SITES];                                   // partial spinors of the four warps
    __shared__ T ss[EPI == EPI_CLOVINV ? 24 : 1][SPLIT_SITES];             // their sum
    __shared__ T sx[EPI == EPI_XPAY ? 24 : 1][SPLIT_SITES];                // the x spinor
    const int w = (int)(threadIdx.x >> 5), q = (int)(threadIdx.x >> 4) & 1, sl = (int)(threadIdx.x & 15);
    const int hh = blockIdx.x * SPLIT_SITES + sl;
    const bool valid = hh < a.Vh;
    const int h = valid ? hh : a.Vh - 1, Vh = a.Vh;
    // |p|^2 enters <p, Ap> only with a shift: decided here, so that a captured launch holds for every shift
    bool with_pnorm = false;
    if constexpr (MODE == CNT_CG_MHAT) with_pnorm = f.scal[S_SIGMA] != 0.0;

    const int xh = h % a.Lxh;
    int r = h / a.Lxh;
    const int y = r % a.L1;
    r /= a.L1;
    const int z = r % a.L2, t = r / a.L2;
    const int sy = a.Lxh, sz = a.Lxh * a.L1, st = sz * a.L2;
    cplx<T> up[3], low[3];
    if (w == 0) {
        const int x = 2 * xh + ((a.parity + y + z + t) & 1);
        const int xf = (x + 1 == a.L0) ? 0 : x + 1, xb = (x == 0) ? a.L0 - 1 : x - 1;
        two_hops<PREC, RECON, DAG, 0>(up, low, a, h, h - xh + (xf >> 1), h - xh + (xb >> 1), q, T(1), T(1));
    } else if (w == 1) {
        two_hops<PREC, RECON, DAG, 1>(up, low, a, h, (y + 1 == a.L1) ? h - (a.L1 - 1) * sy : h + sy,
                                      (y == 0) ? h + (a.L1 - 1) * sy : h - sy, q, T(1), T(1));
    } else if (w == 2) {
        two_hops<PREC, RECON, DAG, 2>(up, low, a, h, (z + 1 == a.L2) ? h - (a.L2 - 1) * sz : h + sz,
                                      (z == 0) ? h + (a.L2 - 1) * sz : h - sz, q, T(1), T(1));
    } else {
        const bool wf = t + 1 == a.L3, wb = t == 0;
        two_hops<PREC, RECON, DAG, 3>(up, low, a, h, wf ? h - (a.L3 - 1) * st : h + st,
                                      wb ? h + (a.L3 - 1) * st : h - st, q, (T)(wf ? a.cf * a.bc : a.cf),
                                      (T)(wb ? a.cb * a.bc : a.cb));
    }
    // this thread's part of the epilogue: part q of components w, w + 4, w + 8
    CloverRow<PREC> row[3];
    if constexpr (EPI != EPI_PLAIN) {
#pragma unroll
        for (int k = 0; k < 3; k++) row[k].load(a.clov, 4 * k + w, h, Vh);
    }
    if constexpr (EPI == EPI_XPAY) {
        const T n = load_scale<PREC>(a.xin, h, Vh);
#pragma unroll
        for (int k = 0; k < 3; k++) {
            const cplx<T> v = load_comp<PREC>(a.xin, 4 * k + w, h, Vh);
            const T e = q ? v.im : v.re;
            sx[2 * (4 * k + w) + q][sl] = PREC == BQ_PREC_HALF ? n * e : e;
        }
    }
    {
        const int ls = w < 2 ? 3 - q : 2 + q;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            sp[w][2 * (3 * q + c)][sl] = up[c].re;
            sp[w][2 * (3 * q + c) + 1][sl] = up[c].im;
            sp[w][2 * (3 * ls + c)][sl] = low[c].re;
            sp[w][2 * (3 * ls + c) + 1][sl] = low[c].im;
        }
    }
    __syncthreads();
    T o[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const int e = 2 * (4 * k + w) + q;
        o[k] = ((sp[0][e][sl] + sp[1][e][sl]) + sp[2][e][sl]) + sp[3][e][sl];
    }
    if constexpr (EPI == EPI_CLOVINV) {
#pragma unroll
        for (int k = 0; k < 3; k++) ss[2 * (4 * k + w) + q][sl] = o[k];
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 3; k++) o[k] = row[k].apply(&ss[0][sl], 4 * k + w, q);
    } else if constexpr (EPI == EPI_XPAY) {
        const T kk = (T)a.k;
#pragma unroll
        for (int k = 0; k < 3; k++) o[k] = fma(-kk, o[k], row[k].apply(&sx[0][sl], 4 * k + w, q));
    }
    if constexpr (MODE != CNT_CG_MHATDAG) {
        if constexpr (PREC == BQ_PREC_HALF) {
            // the site's scale needs all 24 reals: through shared memory (the partial spinors are used up)
            __syncthreads();
#pragma unroll
            for (int k = 0; k < 3; k++) sp[0][2 * (4 * k + w) + q][sl] = o[k];
            __syncthreads();
            if (threadIdx.x < 3 * SPLIT_SITES && valid) {
                const int k = threadIdx.x / SPLIT_SITES;
                T m = 0;
#pragma unroll
                for (int e = 0; e < 24; e++) m = fmaxf(m, fabsf(sp[0][e][sl]));
                const T inv = m > 0 ? 1.0f / m : 0.f;
                uint4 v;
                v.x = f2h(sp[0][8 * k][sl] * inv, sp[0][8 * k + 1][sl] * inv);
                v.y = f2h(sp[0][8 * k + 2][sl] * inv, sp[0][8 * k + 3][sl] * inv);
                v.z = f2h(sp[0][8 * k + 4][sl] * inv, sp[0][8 * k + 5][sl] * inv);
                v.w = f2h(sp[0][8 * k + 6][sl] * inv, sp[0][8 * k + 7][sl] * inv);
                uint4 *p = static_cast<uint4 *>(a.out);
                p[(size_t)k * Vh + h] = v;
                if (k == 0) reinterpret_cast<float *>(p + (size_t)3 * Vh)[h] = m;
            }
        } else if (valid) {
            T *p = static_cast<T *>(a.out);
#pragma unroll
            for (int k = 0; k < 3; k++) p[real_at<T>(4 * k + w, q, h, Vh)] = o[k];
        }
    }
    if constexpr (MODE != 0) {
        constexpr int NV = MODE == CNT_CG_MHAT ? 2 : 1;
        T v[NV];
#pragma unroll
        for (int k = 0; k < NV; k++) v[k] = T(0);
        if (MODE == CNT_CG_MHAT && valid) {
#pragma unroll
            for (int k = 0; k < 3; k++) {
                v[0] = fma(o[k], o[k], v[0]);
                if (with_pnorm) {
                    const T x = sx[2 * (4 * k + w) + q][sl];
                    v[NV - 1] = fma(x, x, v[NV - 1]);
                }
            }
        } else if (MODE == CNT_CG_MHATDAG && valid) {
            const T alpha = (T)f.scal[S_ALPHA], sigma = (T)f.scal[S_SIGMA];
            const T n = load_scale<PREC>(f.p, h, Vh);
            T *xs = static_cast<T *>(f.xs), *rs = static_cast<T *>(f.rs);
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const cplx<T> pc = load_comp<PREC>(f.p, 4 * k + w, h, Vh);
                const T p = (q ? pc.im : pc.re) * n;
                const size_t at = real_at<T>(4 * k + w, q, h, Vh);
                const T rv = fma(-alpha, fma(sigma, p, o[k]), rs[at]);
                xs[at] = fma(alpha, p, xs[at]);
                rs[at] = rv;
                v[0] = fma(rv, rv, v[0]);
            }
        }
        __shared__ T ws[NV][4];
#pragma unroll
        for (int k = 0; k < NV; k++) {
            T s = v[k];
#pragma unroll
            for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
            if ((threadIdx.x & 31) == 0) ws[k][w] = s;
        }
        __syncthreads();
        // one partial per block; the last block to finish sums them in block order and sets the
        // solver scalars (at a few hundred blocks its ticket costs about a microsecond, a separate
        // one-block kernel three)
        __shared__ bool last;
        if (threadIdx.x == 0) {
#pragma unroll
            for (int k = 0; k < NV; k++)
                f.partials[k * gridDim.x + blockIdx.x] = (double)(((ws[k][0] + ws[k][1]) + ws[k][2]) + ws[k][3]);
            __threadfence();
            last = atomicAdd(f.ticket, 1u) == gridDim.x - 1;
        }
        __syncthreads();
        if (!last) return;
        __threadfence();
        double tot[NV];
#pragma unroll
        for (int k = 0; k < NV; k++) tot[k] = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += 128)
#pragma unroll
            for (int k = 0; k < NV; k++) tot[k] += __ldcg(f.partials + k * gridDim.x + i);
        block_sum(tot);
        if (threadIdx.x == 0) {
            *f.ticket = 0;
            if constexpr (MODE == CNT_CG_MHAT) cg_set_alpha(f.scal, tot[0], tot[NV - 1]);
            else cg_set_beta(f.scal, tot[0]);
        }
    }
}

template <int PREC, int RECON>
void launch_pr(const DslashArgs &a, const CgFuse &f, bool dag, int epi, int mode, unsigned grid, cudaStream_t s) {
    if (mode == CNT_CG_MHAT) bq_launch(k_dslash_split<PREC, RECON, false, EPI_XPAY, CNT_CG_MHAT>, grid, 128, s, a, f);
    else if (mode == CNT_CG_MHATDAG) bq_launch(k_dslash_split<PREC, RECON, true, EPI_XPAY, CNT_CG_MHATDAG>, grid, 128, s, a, f);
    else if (dag && epi == EPI_PLAIN) bq_launch(k_dslash_split<PREC, RECON, true, EPI_PLAIN, 0>, grid, 128, s, a, f);
    else if (dag && epi == EPI_CLOVINV) bq_launch(k_dslash_split<PREC, RECON, true, EPI_CLOVINV, 0>, grid, 128, s, a, f);
    else if (dag) bq_launch(k_dslash_split<PREC, RECON, true, EPI_XPAY, 0>, grid, 128, s, a, f);
    else if (epi == EPI_PLAIN) bq_launch(k_dslash_split<PREC, RECON, false, EPI_PLAIN, 0>, grid, 128, s, a, f);
    else if (epi == EPI_CLOVINV) bq_launch(k_dslash_split<PREC, RECON, false, EPI_CLOVINV, 0>, grid, 128, s, a, f);
    else bq_launch(k_dslash_split<PREC, RECON, false, EPI_XPAY, 0>, grid, 128, s, a, f);
}

// FP64 storage on the FP64 units, lattices that fill the chip: two threads per site (lanes
// l and l + 16 of a warp of 16 sites), each with its half spinor through all eight hops,
// then the chirality block q of the clover term: 558 FP64 instructions per thread, 108
// registers, no spills.
template <bool DAG, int EPI>
__global__ void __launch_bounds__(32) k_dslash_pair64(const DslashArgs a) {
    constexpr int P = BQ_PREC_DOUBLE;
    constexpr int SF = DAG ? +1 : -1;
    bq_pdl_enter();
    const int q = (int)(threadIdx.x >> 4) & 1;
    const int hh = (a.rev ? gridDim.x - 1 - blockIdx.x : blockIdx.x) * SPLIT_SITES + (int)(threadIdx.x & 15);
    const bool valid = hh < a.Vh;
    const int h = valid ? hh : a.Vh - 1, Vh = a.Vh;
    const int xh = h % a.Lxh;
    int r = h / a.Lxh;
    const int y = r % a.L1;
    r /= a.L1;
    const int z = r % a.L2, t = r / a.L2;
    const int x = 2 * xh + ((a.parity + y + z + t) & 1);
    const int sy = a.Lxh, sz = a.Lxh * a.L1, st = sz * a.L2;
    const char *Lo = a.links + (size_t)a.parity * 4 * a.lblk;
    const char *Li = a.links + (size_t)(1 - a.parity) * 4 * a.lblk;
    const bool wf = t + 1 == a.L3, wb = t == 0;
    // lowa: the x and y hops' part of spin 3 - q; lowb: the z and t hops' part of spin 2 + q
    cplx<double> up[3], lowa[3], lowb[3];
    int hn = h - xh + (((x + 1 == a.L0) ? 0 : x + 1) >> 1);
    half_hop<P, 18, 0, SF, false, true, true>(up, lowa, a.in, hn, Lo, h, Vh, q, 1.0);
    hn = h - xh + (((x == 0) ? a.L0 - 1 : x - 1) >> 1);
    half_hop<P, 18, 0, -SF, true, false, false>(up, lowa, a.in, hn, Li, hn, Vh, q, 1.0);
    hn = (y + 1 == a.L1) ? h - (a.L1 - 1) * sy : h + sy;
    half_hop<P, 18, 1, SF, false, false, false>(up, lowa, a.in, hn, Lo + a.lblk, h, Vh, q, 1.0);
    hn = (y == 0) ? h + (a.L1 - 1) * sy : h - sy;
    half_hop<P, 18, 1, -SF, true, false, false>(up, lowa, a.in, hn, Li + a.lblk, hn, Vh, q, 1.0);
    hn = (z + 1 == a.L2) ? h - (a.L2 - 1) * sz : h + sz;
    half_hop<P, 18, 2, SF, false, false, true>(up, lowb, a.in, hn, Lo + 2 * a.lblk, h, Vh, q, 1.0);
    hn = (z == 0) ? h + (a.L2 - 1) * sz : h - sz;
    half_hop<P, 18, 2, -SF, true, false, false>(up, lowb, a.in, hn, Li + 2 * a.lblk, hn, Vh, q, 1.0);
    hn = wf ? h - (a.L3 - 1) * st : h + st;
    half_hop<P, 18, 3, SF, false, false, false>(up, lowb, a.in, hn, Lo + 3 * a.lblk, h, Vh, q, wf ? a.cf * a.bc : a.cf);
    hn = wb ? h + (a.L3 - 1) * st : h - st;
    half_hop<P, 18, 3, -SF, true, false, false>(up, lowb, a.in, hn, Li + 3 * a.lblk, hn, Vh, q, wb ? a.cb * a.bc : a.cb);
    // lane 0 of the pair takes spins 0 and 1, lane 1 spins 2 and 3
    cplx<double> o[6];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const double ur = __shfl_xor_sync(0xffffffffu, up[c].re, 16), ui = __shfl_xor_sync(0xffffffffu, up[c].im, 16);
        const double ar = __shfl_xor_sync(0xffffffffu, lowa[c].re, 16), ai = __shfl_xor_sync(0xffffffffu, lowa[c].im, 16);
        const double br = __shfl_xor_sync(0xffffffffu, lowb[c].re, 16), bi = __shfl_xor_sync(0xffffffffu, lowb[c].im, 16);
        o[c] = q ? cplx<double>{lowa[c].re + br, lowa[c].im + bi} : up[c];
        o[3 + c] = q ? cplx<double>{lowb[c].re + ar, lowb[c].im + ai} : cplx<double>{ur, ui};
    }
    if constexpr (EPI != EPI_PLAIN) {
        double d[6];
        cplx<double> m[15], v[6];
        CloverIO<P>::load_block(d, m, a.clov, q, h, Vh);
        if constexpr (EPI == EPI_CLOVINV) {
            herm6_apply(d, m, o, v);
#pragma unroll
            for (int c = 0; c < 6; c++) o[c] = v[c];
        } else {
            cplx<double> xv[6];
#pragma unroll
            for (int c = 0; c < 6; c++) xv[c] = load_comp<P>(a.xin, 6 * q + c, h, Vh);
            herm6_apply(d, m, xv, v);
#pragma unroll
            for (int c = 0; c < 6; c++) o[c] = {fma(-a.k, o[c].re, v[c].re), fma(-a.k, o[c].im, v[c].im)};
        }
    }
    if (!valid) return;
    double2 *po = static_cast<double2 *>(a.out) + (size_t)(6 * q) * Vh + h;
#pragma unroll
    for (int c = 0; c < 6; c++) po[(size_t)c * Vh] = make_double2(o[c].re, o[c].im);
}

}  // namespace

void bq_pair64_launch(const DslashArgs &a, bool dag, int epi, cudaStream_t s) {
    const unsigned grid = bq_split_grid(a.Vh);
    if (dag && epi == EPI_PLAIN) bq_launch(k_dslash_pair64<true, EPI_PLAIN>, grid, 32, s, a);
    else if (dag && epi == EPI_CLOVINV) bq_launch(k_dslash_pair64<true, EPI_CLOVINV>, grid, 32, s, a);
    else if (dag) bq_launch(k_dslash_pair64<true, EPI_XPAY>, grid, 32, s, a);
    else if (epi == EPI_PLAIN) bq_launch(k_dslash_pair64<false, EPI_PLAIN>, grid, 32, s, a);
    else if (epi == EPI_CLOVINV) bq_launch(k_dslash_pair64<false, EPI_CLOVINV>, grid, 32, s, a);
    else bq_launch(k_dslash_pair64<false, EPI_XPAY>, grid, 32, s, a);
}

unsigned bq_split_grid(int Vh) { return (unsigned)((Vh + SPLIT_SITES - 1) / SPLIT_SITES); }

void bq_split_launch(int prec, int recon, const DslashArgs &a, const CgFuse &f, bool dag, int epi, int mode,
                     cudaStream_t s) {
    const unsigned grid = bq_split_grid(a.Vh);
    if (prec == BQ_PREC_DOUBLE) {
        launch_pr<BQ_PREC_DOUBLE, 18>(a, f, dag, epi, mode, grid, s);
    } else if (prec == BQ_PREC_SINGLE) {
        if (recon == 12) launch_pr<BQ_PREC_SINGLE, 12>(a, f, dag, epi, mode, grid, s);
        else if (recon == 8) launch_pr<BQ_PREC_SINGLE, 8>(a, f, dag, epi, mode, grid, s);
        else launch_pr<BQ_PREC_SINGLE, 18>(a, f, dag, epi, mode, grid, s);
    } else {
        if (recon == 12) launch_pr<BQ_PREC_HALF, 12>(a, f, dag, epi, mode, grid, s);
        else if (recon == 8) launch_pr<BQ_PREC_HALF, 8>(a, f, dag, epi, mode, grid, s);
        else launch_pr<BQ_PREC_HALF, 18>(a, f, dag, epi, mode, grid, s);
    }
}
