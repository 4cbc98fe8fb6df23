// bq_gauge.cu -- gauge-side setup steps that precede a solve in the HMC:
//   * stout smearing of the hopping-term links (Section 2, QCD+QED: the
//     fermion action of Eq. 5 hops with singly iterated stout links Ũ), after
//     Morningstar and Peardon, Phys. Rev. D 69 (2004) 054501;
//   * log det A of the clover term (Eq. 2) on one parity, the even-odd
//     preconditioned action's log det A_oo term.
#include <math.h>

#include "bq_geo.cuh"
#include "bq_nvtx.cuh"
#include "bq_reduce.cuh"

// exp(X) of a traceless anti-Hermitian 3x3 matrix: scaling and squaring of a
// degree-14 Taylor polynomial (Moler and Van Loan, "Nineteen dubious ways to
// compute the exponential of a matrix", method 3). X is halved until its
// Frobenius norm is <= 1/2, where the truncation error is below 3e-17.
__device__ M3 expm_su3(const M3 &X) {
    double n2 = 0.0;
    for (int k = 0; k < 9; k++) n2 += X.a[k].re * X.a[k].re + X.a[k].im * X.a[k].im;
    int s = 0;
    double scale = 1.0;
    while (n2 * scale * scale > 0.25 && s < 40) {
        scale *= 0.5;
        s++;
    }
    M3 Y;
    for (int k = 0; k < 9; k++) Y.a[k] = cscale(scale, X.a[k]);
    // Horner: E = I + Y/1 (I + Y/2 (I + ... (I + Y/14)))
    M3 E;
    for (int k = 0; k < 9; k++) E.a[k] = {(k % 4 == 0) ? 1.0 : 0.0, 0.0};
    for (int j = 14; j >= 1; j--) {
        M3 T = mmul(Y, E);
        for (int k = 0; k < 9; k++) {
            E.a[k] = cscale(1.0 / j, T.a[k]);
            if (k % 4 == 0) E.a[k].re += 1.0;
        }
    }
    for (int q = 0; q < s; q++) E = mmul(E, E);
    return E;
}

// exp(X) = exp(iQ), Q = -iX Hermitian traceless, in closed form by the
// Cayley-Hamilton theorem (Morningstar and Peardon 2004, Section III):
// exp(iQ) = f0 + f1 Q + f2 Q^2 with the f_j from c0 = det Q = tr Q^3 / 3 and
// c1 = tr Q^2 / 2. For c0 < 0 the f_j of -c0 are used, f_j(-c0) = (-1)^j
// conj(f_j(c0)), which keeps the angle theta in [0, pi/2] and the denominator
// 9u^2 - w^2 >= 2 c1 away from zero; c1 ~ 0 (Q ~ 0) takes the Taylor path.
__device__ M3 expm_su3_ch(const M3 &X) {
    M3 Q;
    for (int k = 0; k < 9; k++) Q.a[k] = {X.a[k].im, -X.a[k].re};  // -i X
    const M3 Q2 = mmul(Q, Q);
    const M3 Q3 = mmul(Q, Q2);
    const double c1 = 0.5 * (Q2.a[0].re + Q2.a[4].re + Q2.a[8].re);
    if (!(c1 > 1e-12)) return expm_su3(X);
    double c0 = (Q3.a[0].re + Q3.a[4].re + Q3.a[8].re) / 3.0;
    const bool neg = c0 < 0.0;
    c0 = fabs(c0);
    const double c0max = 2.0 * pow(c1 / 3.0, 1.5);
    const double theta = acos(fmin(c0 / c0max, 1.0));
    const double u = sqrt(c1 / 3.0) * cos(theta / 3.0);
    const double w = sqrt(c1) * sin(theta / 3.0);
    const double w2 = w * w, u2 = u * u;
    // xi0(w) = sin(w) / w, by its series near w = 0
    const double xi0 = (fabs(w) < 0.05) ? 1.0 - w2 / 6.0 * (1.0 - w2 / 20.0 * (1.0 - w2 / 42.0)) : sin(w) / w;
    const double cw = cos(w);
    const cplx<double> e2iu = {cos(2.0 * u), sin(2.0 * u)}, emiu = {cos(u), -sin(u)};
    // h0 = (u^2 - w^2) e^{2iu} + e^{-iu} [8 u^2 cos w + 2 i u (3u^2 + w^2) xi0]
    cplx<double> h0 = cadd(cscale(u2 - w2, e2iu), cmul(emiu, cplx<double>{8.0 * u2 * cw, 2.0 * u * (3.0 * u2 + w2) * xi0}));
    // h1 = 2u e^{2iu} - e^{-iu} [2u cos w - i (3u^2 - w^2) xi0]
    cplx<double> h1 = csub(cscale(2.0 * u, e2iu), cmul(emiu, cplx<double>{2.0 * u * cw, -(3.0 * u2 - w2) * xi0}));
    // h2 = e^{2iu} - e^{-iu} [cos w + 3 i u xi0]
    cplx<double> h2 = csub(e2iu, cmul(emiu, cplx<double>{cw, 3.0 * u * xi0}));
    const double inv = 1.0 / (9.0 * u2 - w2);
    h0 = cscale(inv, h0);
    h1 = cscale(inv, h1);
    h2 = cscale(inv, h2);
    if (neg) {  // f_j(-c0) = (-1)^j conj(f_j(c0))
        h0 = cconj(h0);
        h1 = cscale(-1.0, cconj(h1));
        h2 = cconj(h2);
    }
    M3 E;
    for (int k = 0; k < 9; k++) E.a[k] = cadd(cmul(h1, Q.a[k]), cmul(h2, Q2.a[k]));
    E.a[0] = cadd(E.a[0], h0);
    E.a[4] = cadd(E.a[4], h0);
    E.a[8] = cadd(E.a[8], h0);
    return E;
}

// f_j of exp(iQ) = f0 + f1 Q + f2 Q^2 by the Taylor series to order N: every power of Q is
// a + b Q + c Q^2 by the Cayley-Hamilton theorem (Q^3 = c1 Q + c0), with real a, b, c of two
// operations per order. Truncation below 1e-17 for eigenvalues up to 0.2 (N = 11) or 1 (N = 18).
template <int N>
__device__ __forceinline__ void exp_coefficients(double c0, double c1, cplx<double> f[3]) {
    double a = 0.0, b = 0.0, c = 1.0;  // Q^2
    f[0] = {1.0, 0.0};
    f[1] = {0.0, 1.0};
    f[2] = {-0.5, 0.0};
    double inv = 0.5;
#pragma unroll
    for (int n = 3; n <= N; n++) {
        const double a1 = c * c0, b1 = n == 3 ? c1 : fma(c, c1, a);  // times Q
        c = b;
        a = a1;
        b = b1;
        inv *= 1.0 / n;
        const double s = (n & 2) ? -inv : inv;  // i^n / n!
        if (n & 1) {
            f[0].im = fma(s, a, f[0].im);
            f[1].im = fma(s, b, f[1].im);
            f[2].im = fma(s, c, f[2].im);
        } else {
            f[0].re = fma(s, a, f[0].re);
            f[1].re = fma(s, b, f[1].re);
            f[2].re = fma(s, c, f[2].re);
        }
    }
}

// exp(X) of a traceless anti-Hermitian X given by its nine reals (imaginary parts of the diagonal,
// the entries 01, 02, 12): the series for eigenvalues up to 1 (2 sqrt(c1 / 3) bounds them), the
// closed form beyond
__device__ __forceinline__ M3 exp_antiherm(const double q[3], const cplx<double> x[3]) {
    // Q = -iX: diagonal q, off-diagonal -i x
    const cplx<double> q01 = {x[0].im, -x[0].re}, q02 = {x[1].im, -x[1].re}, q12 = {x[2].im, -x[2].re};
    const double n01 = fma(q01.re, q01.re, q01.im * q01.im), n02 = fma(q02.re, q02.re, q02.im * q02.im),
                 n12 = fma(q12.re, q12.re, q12.im * q12.im);
    const double c1 = fma(0.5, fma(q[0], q[0], fma(q[1], q[1], q[2] * q[2])), n01 + n02 + n12);
    if (!(c1 <= 0.75)) {
        M3 X;
        for (int k = 0; k < 3; k++) X.a[4 * k] = {0.0, q[k]};
        for (int e = 0; e < 3; e++) {
            const int i = e < 2 ? 0 : 1, j = e == 0 ? 1 : 2;
            X.a[i * 3 + j] = x[e];
            X.a[j * 3 + i] = {-x[e].re, x[e].im};
        }
        return expm_su3_ch(X);
    }
    // c0 = det Q
    const cplx<double> t = cmul(q01, q12);
    const double c0 = q[0] * fma(q[1], q[2], -n12) - fma(q[2], n01, q[1] * n02) +
                      2.0 * fma(t.re, q02.re, t.im * q02.im);
    cplx<double> f[3];
    if (c1 <= 0.03) exp_coefficients<11>(c0, c1, f);
    else exp_coefficients<18>(c0, c1, f);
    // Q^2: diagonal, then 01 = q01 (q0 + q1) + q02 conj(q12), 02 = q02 (q0 + q2) + q01 q12,
    // 12 = q12 (q1 + q2) + conj(q01) q02
    const double s0 = fma(q[0], q[0], n01 + n02), s1 = fma(q[1], q[1], n01 + n12), s2 = fma(q[2], q[2], n02 + n12);
    const cplx<double> z01 = cfmac(q12, q02, cscale(q[0] + q[1], q01));
    const cplx<double> z02 = cfma(q01, q12, cscale(q[0] + q[2], q02));
    const cplx<double> z12 = cfmac(q01, q02, cscale(q[1] + q[2], q12));
    M3 E;
    E.a[0] = {fma(f[2].re, s0, fma(f[1].re, q[0], f[0].re)), fma(f[2].im, s0, fma(f[1].im, q[0], f[0].im))};
    E.a[4] = {fma(f[2].re, s1, fma(f[1].re, q[1], f[0].re)), fma(f[2].im, s1, fma(f[1].im, q[1], f[0].im))};
    E.a[8] = {fma(f[2].re, s2, fma(f[1].re, q[2], f[0].re)), fma(f[2].im, s2, fma(f[1].im, q[2], f[0].im))};
    E.a[1] = cfma(f[2], z01, cmul(f[1], q01));
    E.a[2] = cfma(f[2], z02, cmul(f[1], q02));
    E.a[5] = cfma(f[2], z12, cmul(f[1], q12));
    E.a[3] = cfma(f[2], cconj(z01), cmul(f[1], cconj(q01)));
    E.a[6] = cfma(f[2], cconj(z02), cmul(f[1], cconj(q02)));
    E.a[7] = cfma(f[2], cconj(z12), cmul(f[1], cconj(q12)));
    return E;
}

// one stout step for every link: C = rho sum_{nu != mu} (upper + lower staple) in double-float,
// Omega = C U^dag, X = traceless anti-Hermitian part of Omega
// (= i Q with Q = (i/2)(Omega^dag - Omega) - (i/6) tr(Omega^dag - Omega)),
// U' = exp(X) U in FP64. Links are periodic in every direction. A block of four warps takes 32
// consecutive sites, warp mu their links U_mu. Bound by the FP64 pipe and the packed FP32 products
// together: about 430 FP64 instructions per link (Omega 90, series and Q^2 140, exp(X) 60, times
// U 108) are 1.9 ms of the 2.45 ms at 24^3x48; three blocks per SM (168 registers).
#ifndef STOUT_MIN_BLOCKS
#define STOUT_MIN_BLOCKS 3
#endif
template <typename LINKS>
__global__ void __launch_bounds__(128, STOUT_MIN_BLOCKS) k_stout_step(double2 *out, const double2 *in, LINKS P, Geo g,
                                                                      double rho) {
    const long long x = (long long)blockIdx.x * 32 + (threadIdx.x & 31);
    const int mu = threadIdx.x >> 5;
    if (x >= g.V) return;
    const long long V = g.V, xpm = lex_step(g, x, mu, +1);
    M3p Cd;
#pragma unroll
    for (int k = 0; k < 9; k++) Cd.hi[k] = Cd.lo[k] = make_float2(0.f, 0.f);
    // the six staples as three-link paths, multiplied out left to right; one copy of the
    // product's code, one partial product and one link live
#pragma unroll 1
    for (int st = 0; st < 6; st++) {
        const int nu = (st >> 1) + ((st >> 1) >= mu ? 1 : 0);  // the three directions other than mu
        const bool lower = st & 1;
        const long long xmn = lex_step(g, x, nu, -1);
        // upper: U_nu(x) U_mu(x+nu) U_nu(x+mu)^dag; lower: U_nu(x-nu)^dag U_mu(x-nu) U_nu(x-nu+mu)
        const long long s1 = lower ? xmn : lex_step(g, x, nu, +1);
        const long long s2 = lower ? lex_step(g, xmn, mu, +1) : xpm;
        M3p A = load_link_pair(P, V, lower ? xmn : x, nu, lower);
#pragma unroll 1
        for (int j = 0; j < 2; j++) mmul_pair(A, load_link_pair(P, V, j ? s2 : s1, j ? nu : mu, j && !lower));
        madd_pair(Cd, A, 1.0f);
    }
    // Omega = C U^dag; X from its anti-Hermitian part (diagonal: imaginary parts only)
    const M3 U = load_link(in, V, x, mu);
    double q[3];
    cplx<double> xo[3];
    {
        M3 C;
#pragma unroll
        for (int k = 0; k < 9; k++)
            C.a[k] = {(double)Cd.hi[k].x + (double)Cd.lo[k].x, (double)Cd.hi[k].y + (double)Cd.lo[k].y};
#pragma unroll
        for (int i = 0; i < 3; i++) {
            double s = 0.0;  // Im sum_k C_ik conj(U_ik)
#pragma unroll
            for (int k = 0; k < 3; k++) s = fma(C.a[i * 3 + k].im, U.a[i * 3 + k].re, fma(-C.a[i * 3 + k].re, U.a[i * 3 + k].im, s));
            q[i] = rho * s;
        }
        const double tr = (q[0] + q[1] + q[2]) * (1.0 / 3.0);
#pragma unroll
        for (int i = 0; i < 3; i++) q[i] -= tr;
#pragma unroll
        for (int e = 0; e < 3; e++) {
            const int i = e < 2 ? 0 : 1, j = e == 0 ? 1 : 2;
            cplx<double> o = {0.0, 0.0}, p = {0.0, 0.0};  // Omega_ij, Omega_ji
#pragma unroll
            for (int k = 0; k < 3; k++) {
                o = cfmac(U.a[j * 3 + k], C.a[i * 3 + k], o);
                p = cfmac(U.a[i * 3 + k], C.a[j * 3 + k], p);
            }
            xo[e] = {0.5 * rho * (o.re - p.re), 0.5 * rho * (o.im + p.im)};
        }
    }
    const M3 Un = mmul(exp_antiherm(q, xo), U);
    double2 *p = out + (long long)mu * 9 * V + x;
    for (int k = 0; k < 9; k++) p[k * V] = make_double2(Un.a[k].re, Un.a[k].im);
}

// A thread reads its own link from `in` and every other one from the split, so that a step may write over its
// input: beside U_hop only the split needs memory. It lies in a field that is out of date, or in what the
// caller lends; else it is allocated for the call, for one step from 2^17 sites on only, where that takes
// less time than splitting each link at its uses (0.15 against 0.19 ms at V = 166 320, 0.1 against 0.02 ms
// at 41 472), and where it does not fit, one step does without.
int bq_prepare_hop_links(bq_ctx *c, float4 *lent) {
    if (c->U_hop_valid) return BQ_OK;
    BqRange range("stout smearing");
    const size_t bytes = (size_t)c->V * 4 * 9 * sizeof(double2);
    BQ_TRY(bq_alloc((void **)&c->U_hop, bytes));
    float4 *own = nullptr;
    PairLinks P = bq_split_place(c, false);
    const bool keep = P.p;
    if (!P.p) P = {lent, 0};
    if (!P.p && (c->stout_iter > 1 || c->V >= (1LL << 17))) {
        const int s = bq_alloc((void **)&own, bytes);
        if (s != BQ_OK && c->stout_iter > 1) return s;
        P.p = own;
    }
    const Geo g = geo_of(c);
    const unsigned grid = grid_for(c->V, 32);
    const double2 *src = c->U_canon;
    int status = BQ_OK;
    for (int it = 0; it < c->stout_iter && status == BQ_OK; it++) {
        if (P.p) {
            status = bq_split_links(c, src, P, keep);
            if (status != BQ_OK) break;
            k_stout_step<<<grid, 128, 0, c->stream>>>(c->U_hop, src, P, g, c->stout_rho);
        } else {
            k_stout_step<<<grid, 128, 0, c->stream>>>(c->U_hop, src, src, g, c->stout_rho);
        }
        if (cudaGetLastError() != cudaSuccess) {
            bq_set_error("stout smearing launch failed");
            status = BQ_ERR_CUDA;
        }
        BQ_COUNT(c);
        src = c->U_hop;
    }
    if (own) {
        cudaStreamSynchronize(c->stream);
        cudaFree(own);
    }
    if (status == BQ_OK) c->U_hop_valid = 1;
    return status;
}

extern "C" int bq_set_stout(bq_ctx *c, double rho, int n_iter) {
    if (!c || !(rho >= 0.0 && rho <= 1.0) || n_iter < 0 || n_iter > 64) {
        bq_set_error("bq_set_stout: need 0 <= rho <= 1 and 0 <= n_iter <= 64");
        return BQ_ERR_ARG;
    }
    if (rho == 0.0) n_iter = 0;
    if (c->stout_iter != n_iter || c->stout_rho != rho) {
        c->stout_iter = n_iter;
        c->stout_rho = rho;
        c->U_hop_valid = 0;
        for (int p = 0; p < BQ_NFIELD; p++) c->links_valid[p] = 0;
    }
    return BQ_OK;
}

extern "C" int bq_get_hop_links(bq_ctx *c, double *U, int where) {
    if (!c || !U || !(where == BQ_HOST || where == BQ_DEVICE)) {
        bq_set_error("bq_get_hop_links: bad arguments");
        return BQ_ERR_ARG;
    }
    if (!c->have_gauge) {
        bq_set_error("gauge field not set");
        return BQ_ERR_STATE;
    }
    const double2 *src = c->U_canon;
    if (c->stout_iter > 0) {
        // device memory that takes the result serves as work space first
        const bool lend = where == BQ_DEVICE && (uintptr_t)U % sizeof(float4) == 0 && bq_links_direct(c, U);
        BQ_TRY(bq_prepare_hop_links(c, lend ? (float4 *)U : nullptr));
        src = c->U_hop;
    }
    return bq_links_out(c, U, src, where);
}

// --------------------------------------------------------------------------
// log det of the clover term on one parity, per site and chirality block, in
// FP64. Sums: [0] log|det|, [1] blocks with det < 0.

// LU with partial pivoting of chirality block b of half-site h: log|det| =
// sum log|pivot|, the sign (real for a Hermitian block) from the pivots'
// phases and the row swaps; -inf for a zero pivot
__device__ __noinline__ double logdet6_pivoted(const double2 *blk, int b, int h, int Vh, bool *negative) {
    cplx<double> B[36];
    load_herm6(blk, b, h, Vh, B);
    double la = 0.0;
    cplx<double> ph = {1.0, 0.0};
    int swaps = 0;
    for (int col = 0; col < 6; col++) {
        int piv = col;
        double best = hypot(B[col * 6 + col].re, B[col * 6 + col].im);
        for (int r = col + 1; r < 6; r++) {
            const double m = hypot(B[r * 6 + col].re, B[r * 6 + col].im);
            if (m > best) {
                best = m;
                piv = r;
            }
        }
        if (!(best > 0.0)) {
            *negative = false;
            return -INFINITY;
        }
        if (piv != col) {
            swaps++;
            for (int j = 0; j < 6; j++) {
                const cplx<double> t = B[col * 6 + j];
                B[col * 6 + j] = B[piv * 6 + j];
                B[piv * 6 + j] = t;
            }
        }
        const cplx<double> p = B[col * 6 + col];
        la += log(best);
        ph = cmul(ph, cplx<double>{p.re / best, p.im / best});
        const double n2 = p.re * p.re + p.im * p.im;
        const cplx<double> inv = {p.re / n2, -p.im / n2};
        for (int r = col + 1; r < 6; r++) {
            const cplx<double> f = cmul(B[r * 6 + col], inv);
            for (int j = col; j < 6; j++) B[r * 6 + j] = csub(B[r * 6 + j], cmul(f, B[col * 6 + j]));
        }
    }
    *negative = ((swaps & 1) ? -ph.re : ph.re) < 0.0;
    return la;
}

// Fast path: A = L D L^dag without pivoting (D real), det A = prod d_j, taken
// when every |d_j| is at least 0.1 of the block's largest entry; otherwise the
// pivoted LU above. Loops of fixed trip count with guards unroll completely,
// so that the block stays in registers.
__global__ void __launch_bounds__(RED_THREADS) k_clover_logdet(const double2 *blk, int Vh, double *partials,
                                                               unsigned int *ticket, double *out) {
    double v[2] = {0.0, 0.0};
    for (int idx = blockIdx.x * blockDim.x + threadIdx.x; idx < 2 * Vh; idx += gridDim.x * blockDim.x) {
        const int h = idx % Vh, b = idx / Vh;
        cplx<double> B[36];
        load_herm6(blk, b, h, Vh, B);
        Ldl6 f;
        const bool fast = f.factor(B);
        double det = 1.0;
#pragma unroll
        for (int j = 0; j < 6; j++) det *= f.d[j];
        bool neg;
        double la;
        if (fast) {
            la = log(fabs(det));
            neg = det < 0.0;
        } else {
            la = logdet6_pivoted(blk, b, h, Vh, &neg);
        }
        v[0] += la;
        v[1] += neg ? 1.0 : 0.0;
    }
    double tot[2];
    if (grid_sum(v, partials, ticket, tot) && threadIdx.x == 0) {
        out[0] = tot[0];
        out[1] = tot[1];
    }
}

extern "C" int bq_clover_logdet(bq_ctx *c, int parity, double *logdet, int *negative) {
    if (!c || !logdet || !(parity == 0 || parity == 1)) {
        bq_set_error("bq_clover_logdet: bad arguments");
        return BQ_ERR_ARG;
    }
    if (!c->have_gauge) {
        bq_set_error("gauge field not set");
        return BQ_ERR_STATE;
    }
    BQ_TRY(bq_prepare_clover(c, BQ_PREC_DOUBLE));
    const size_t pblk = (size_t)36 * c->Vh;
    const double2 *blk = reinterpret_cast<const double2 *>(c->clov_master) + (size_t)(parity * 2 + 0) * pblk;
    double *res = c->red_partials + 2 * RED_MAX_BLOCKS;
    k_clover_logdet<<<red_grid(2 * c->Vh), RED_THREADS, 0, c->stream>>>(blk, c->Vh, c->red_partials, c->red_ticket,
                                                                          res);
    BQ_LAUNCH_CHECK();
    BQ_COUNT(c);
    double h[2];
    BQ_CUDA_TRY(cudaMemcpyAsync(h, res, sizeof h, cudaMemcpyDeviceToHost, c->stream));
    BQ_CUDA_TRY(cudaStreamSynchronize(c->stream));
    *logdet = h[0];
    if (negative) *negative = (int)h[1];
    if (!(h[0] > -INFINITY)) {
        bq_set_error("bq_clover_logdet: singular clover block");
        return BQ_ERR_CLOVER_SINGULAR;
    }
    return BQ_OK;
}
