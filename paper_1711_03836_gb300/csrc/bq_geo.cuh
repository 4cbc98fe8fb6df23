// bq_geo.cuh -- full-lattice geometry and FP64 3x3 complex matrix helpers
// shared by the setup kernels (link packing, clover build, stout smearing).
#pragma once

#include "bq_internal.cuh"
#include "bq_pairs.cuh"

struct Geo {
    int L0, L1, L2, L3;
    long long V;
    int Vh;
};

__device__ __forceinline__ void lex_coords(const Geo &g, long long lex, int c[4]) {
    c[0] = (int)(lex % g.L0);
    lex /= g.L0;
    c[1] = (int)(lex % g.L1);
    lex /= g.L1;
    c[2] = (int)(lex % g.L2);
    c[3] = (int)(lex / g.L2);
}
__device__ __forceinline__ long long lex_of(const Geo &g, const int c[4]) {
    return c[0] + (long long)g.L0 * (c[1] + (long long)g.L1 * (c[2] + (long long)g.L2 * c[3]));
}
__device__ __forceinline__ long long lex_step(const Geo &g, long long lex, int mu, int dir) {
    int c[4];
    lex_coords(g, lex, c);
    const int Ls[4] = {g.L0, g.L1, g.L2, g.L3};
    c[mu] += dir;
    if (c[mu] < 0) c[mu] += Ls[mu];
    if (c[mu] >= Ls[mu]) c[mu] -= Ls[mu];
    return lex_of(g, c);
}

static inline Geo geo_of(const bq_ctx *c) { return Geo{c->L[0], c->L[1], c->L[2], c->L[3], c->V, c->Vh}; }

static inline unsigned grid_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

struct M3 {
    cplx<double> a[9];
};

// gauge links inside the library: element k of U_mu(lex) at (mu * 9 + k) * V + lex, so that the
// threads of a warp (consecutive sites) read consecutive addresses
__device__ __forceinline__ M3 load_link(const double2 *U, long long V, long long lex, int mu) {
    M3 m;
    const double2 *p = U + (long long)mu * 9 * V + lex;
    for (int k = 0; k < 9; k++) {
        const double2 v = p[k * V];
        m.a[k] = {v.x, v.y};
    }
    return m;
}
__device__ __forceinline__ M3 mmul(const M3 &x, const M3 &y) {
    M3 m;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) {
            cplx<double> s = {0, 0};
            for (int k = 0; k < 3; k++) s = cfma(x.a[i * 3 + k], y.a[k * 3 + j], s);
            m.a[i * 3 + j] = s;
        }
    return m;
}


// write a Hermitian 6x6 (given as full matrix) into packed FP64 storage of one block
__device__ __forceinline__ void store_herm6(double2 *blk, int b, int h, int Vh, const cplx<double> B[36]) {
    double2 *p = blk + (size_t)(18 * b) * Vh + h;
    for (int k = 0; k < 3; k++) p[(size_t)k * Vh] = make_double2(B[(2 * k) * 7].re, B[(2 * k + 1) * 7].re);
    int k = 0;
    for (int i = 0; i < 6; i++)
        for (int j = i + 1; j < 6; j++) {
            p[(size_t)(3 + k) * Vh] = make_double2(B[i * 6 + j].re, B[i * 6 + j].im);
            k++;
        }
}
__device__ __forceinline__ void load_herm6(const double2 *blk, int b, int h, int Vh, cplx<double> B[36]) {
    const double2 *p = blk + (size_t)(18 * b) * Vh + h;
    for (int k = 0; k < 3; k++) {
        double2 v = p[(size_t)k * Vh];
        B[(2 * k) * 7] = {v.x, 0.0};
        B[(2 * k + 1) * 7] = {v.y, 0.0};
    }
    int k = 0;
    for (int i = 0; i < 6; i++)
        for (int j = i + 1; j < 6; j++) {
            double2 v = p[(size_t)(3 + k) * Vh];
            B[i * 6 + j] = {v.x, v.y};
            B[j * 6 + i] = {v.x, -v.y};
            k++;
        }
}


// c - a b and c - a conj(b), one FMA per real product
__device__ __forceinline__ cplx<double> cfnma(cplx<double> a, cplx<double> b, cplx<double> c) {
    return {fma(-a.re, b.re, fma(a.im, b.im, c.re)), fma(-a.re, b.im, fma(-a.im, b.re, c.im))};
}
__device__ __forceinline__ cplx<double> cfnmac(cplx<double> a, cplx<double> b, cplx<double> c) {
    return {fma(-a.re, b.re, fma(-a.im, b.im, c.re)), fma(a.re, b.im, fma(-a.im, b.re, c.im))};
}

// B = L D L^dag of a Hermitian 6x6 block without pivoting (L unit lower triangular, D real): false
// unless every |d_j| is at least 0.1 of the block's largest entry (compared as squares: 36 hypot calls
// took a third of the inverse's FP64 time; a block whose squares leave the double range is refused
// here and takes the pivoted path). The loops run over fixed trip counts with guards, so that they
// unroll completely and every array stays in registers. W_ik = L_ik d_k.
struct Ldl6 {
    cplx<double> L[36];
    double d[6], dinv[6];
    __device__ __forceinline__ bool factor(const cplx<double> B[36]) {
        double s2 = 0.0;
#pragma unroll
        for (int i = 0; i < 6; i++)
#pragma unroll
            for (int j = 0; j < 6; j++)
                if (j >= i) {
                    const cplx<double> v = B[i * 6 + j];
                    s2 = fmax(s2, i == j ? v.re * v.re : fma(v.re, v.re, v.im * v.im));
                }
        bool ok = s2 > 1e-280 && s2 < 1e280;
        cplx<double> W[36];
#pragma unroll
        for (int j = 0; j < 6; j++) {
            double dj = B[j * 7].re;
#pragma unroll
            for (int k = 0; k < 6; k++)
                if (k < j) dj = fma(-W[j * 6 + k].re, L[j * 6 + k].re, fma(-W[j * 6 + k].im, L[j * 6 + k].im, dj));
            ok = ok && dj * dj >= 0.01 * s2;
            d[j] = dj;
            dinv[j] = 1.0 / dj;
#pragma unroll
            for (int i = 0; i < 6; i++)
                if (i > j) {
                    cplx<double> t = B[i * 6 + j];
#pragma unroll
                    for (int k = 0; k < 6; k++)
                        if (k < j) t = cfnmac(W[i * 6 + k], L[j * 6 + k], t);
                    W[i * 6 + j] = t;
                    L[i * 6 + j] = cscale(dinv[j], t);
                }
        }
        return ok;
    }
};

// 3x3 complex matrices in double-float: GB300 runs FP32 at ~60x its FP64 rate, and the staple
// and clover-leaf products are most of the work of a stout step and of the clover build. An
// entry is a (re, im) pair of leading parts and one of low parts, and the products run on such
// pairs with the packed FP32 instructions (one instruction for both components), each entry a
// lazy sum of six products. The links come split (k_split_links, same order as the master
// field, float4 (re.hi, im.hi, re.lo, im.lo)): splitting the doubles at every use took a
// quarter of the instructions, and reading [site][4][9] links one site per thread 8 times the
// L1 wavefronts. Against scalar sums on links split at each use (24^3x48, V = 663 552): clover
// build 5.86 -> 2.30 ms (with ten products per plane instead of twelve), stout step
// 5.79 -> 2.45 ms (with the exponential's series); the packed FP32 work is 1.4 ms of the first.
struct M3p {
    float2 hi[9], lo[9];
};
// a link entry as (re.hi, im.hi, re.lo, im.lo), exactly but for the last five bits of the low parts;
// normalised, so that the products of two low parts which the sums leave out are below 2^-50 of a
// term and of either sign (the truncating split alone leaves 2^-48, all of one sign)
__device__ __forceinline__ float4 split_entry(double2 v) {
    const df a = normalise(df_from_double(v.x)), b = normalise(df_from_double(v.y));
    return make_float4(a.hi, b.hi, a.lo, b.lo);
}
// the links of one direction: split beforehand, or split at each use where there was no memory to hold that
__device__ __forceinline__ const float4 *links_of(const PairLinks &P, long long V, int mu) {
    return P.p + (long long)mu * 9 * V + (mu >= 2 ? P.gap : 0);
}
__device__ __forceinline__ const double2 *links_of(const double2 *U, long long V, int mu) {
    return U + (long long)mu * 9 * V;
}
__device__ __forceinline__ float4 split_entry(float4 v) { return v; }
// U_mu(lex), or its adjoint
template <typename LINKS>
__device__ __forceinline__ M3p load_link_pair(const LINKS &P, long long V, long long lex, int mu, bool dag) {
    M3p m;
    const auto *p = links_of(P, V, mu) + lex;
    const float sg = dag ? -1.0f : 1.0f;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const float4 v = split_entry(p[(dag ? j * 3 + i : i * 3 + j) * V]);
            m.hi[i * 3 + j] = make_float2(v.x, sg * v.y);
            m.lo[i * 3 + j] = make_float2(v.z, sg * v.w);
        }
    return m;
}
__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 swap2(float2 a) { return make_float2(a.y, a.x); }
// x = x y, row by row
__device__ __forceinline__ void mmul_pair(M3p &x, const M3p &y) {
#pragma unroll
    for (int i = 0; i < 3; i++) {
        float2 rh[3], rl[3];
#pragma unroll
        for (int j = 0; j < 3; j++) {
            dfsum2 z;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                const float2 wh = x.hi[i * 3 + k], wl = x.lo[i * 3 + k], h = y.hi[k * 3 + j], l = y.lo[k * 3 + j];
                if (k == 0) z = dfs2_prod(dup(wh.x), dup(wl.x), h, l);
                else dfs2_add_prod(z, dup(wh.x), dup(wl.x), h, l);
                dfs2_add_prod(z, make_float2(-wh.y, wh.y), make_float2(-wl.y, wl.y), swap2(h), swap2(l));
            }
            dfs2_done(z, rh[j], rl[j]);
        }
#pragma unroll
        for (int j = 0; j < 3; j++) {
            x.hi[i * 3 + j] = rh[j];
            x.lo[i * 3 + j] = rl[j];
        }
    }
}
// x = s x + y (s = +-1), normalised: a low part above half an ulp of its leading part would lose
// the product of two low parts in the multiplication that follows
__device__ __forceinline__ void madd_pair(M3p &x, const M3p &y, float s) {
#pragma unroll
    for (int k = 0; k < 9; k++) {
        const float2 a = __fmul2_rn(dup(s), x.hi[k]), al = __fmul2_rn(dup(s), x.lo[k]);
        const dfsum2 t = two_sum2(a, y.hi[k]);
        dfs2_done({t.s, __fadd2_rn(t.c, __fadd2_rn(al, y.lo[k]))}, x.hi[k], x.lo[k]);
    }
}
