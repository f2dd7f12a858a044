// Molecular-dynamics forces and the leapfrog step of the two-flavour HMC
// (Sec. 2, Eq. 4), FP64.
//
// A link moves along U_mu(x) -> exp(eps T_a) U_mu(x), T_a = i lambda_a / 2
// (Gell-Mann matrices); a gradient is dS/d eps per link and generator, stored
// g[site][mu][a] (lexicographic sites, the MD force is its negative).  Every
// kernel gathers what one link receives (one thread per link, no atomics):
//
//   hops     D holds U_mu(x) in the forward hop out of x and, as U^dag, in
//            the backward hop into x + mu, so
//              Re <Y, dD X> = Re tr(T_a M),
//              M = -1/2 s U B1 + 1/2 s B2 U^dag,
//            B1 = sum_s [(1 - g_mu) X(x+mu)]_s Y(x)_s^dag,
//            B2 = sum_s [(1 + g_mu) X(x)]_s Y(x+mu)_s^dag (colour outer
//            products), s the antiperiodic time sign of the link;
//   clover   the term c_sw (i/4) sigma_{rho sigma} Fhat_{rho sigma}(y) with
//            Fhat = (Q - Q^dag)/8 and Q the four leaves at y: per site and
//            plane Lam[k][i] = (i/4) sum_ab sigma_ab M_{(b k),(a i)}, with
//            M = X Y^dag (pseudofermion) or M = A(y)^-1 (log det), and
//            Om = Lam - Lam^dag; a leaf f0 f1 f2 f3 whose factor f_j is the
//            link contributes (c_sw / 8) U B Om A for f_j = U and
//            -(c_sw / 8) B Om A U^dag for f_j = U^dag, A = f0..f_{j-1},
//            B = f_{j+1}..f3 (summed as in k_force_clover);
//   gauge    S_g = beta sum_P (1 - Re tr U_P / 3): M = -(beta / 3) U sum
//            (staples).
//
// Re tr(T_a M) = -Re tr(T_a M^dag) for the anti-Hermitian T_a, so a term that
// ends in U^dag is traded for minus its adjoint, and every kernel collects one
// matrix W with M = U W.
//
// The kernels are bound by GB300's FP64 pipe (2 multiply-adds per clock and
// SM), not by their loads: what counts is the number of 3x3 products per link.
// A block works on links of one direction and parity at consecutive ranks, so
// directions never diverge within a warp and the link loads are coalesced.
//
// The leapfrog step (p -= dt/2 g; U <- exp(dt P) U; p -= dt/2 g, with
// P = sum_a p^a T_a) exponentiates with a Taylor series after scaling and
// squaring (Moler & Van Loan, "Nineteen dubious ways to compute the
// exponential of a matrix, twenty-five years later", 2003).
#include <cmath>
#include <vector>

#include "lqcd_internal.cuh"

namespace {

using Cd = cx<double>;

struct M3 {
    Cd m[3][3];
};

__device__ __forceinline__ M3 m3_zero()
{
    M3 c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) c.m[i][j] = mk(0.0, 0.0);
    return c;
}
__device__ __forceinline__ M3 m3_one()
{
    M3 c = m3_zero();
#pragma unroll
    for (int i = 0; i < 3; i++) c.m[i][i] = mk(1.0, 0.0);
    return c;
}
// acc += a b, every product entering its sum through a fused multiply-add
__device__ __forceinline__ void mul_add(M3 &acc, const M3 &a, const M3 &b)
{
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            double re = acc.m[i][j].re, im = acc.m[i][j].im;
#pragma unroll
            for (int k = 0; k < 3; k++) {
                re = fmx(a.m[i][k].re, b.m[k][j].re, re);
                re = fmx(-a.m[i][k].im, b.m[k][j].im, re);
                im = fmx(a.m[i][k].re, b.m[k][j].im, im);
                im = fmx(a.m[i][k].im, b.m[k][j].re, im);
            }
            acc.m[i][j] = mk(re, im);
        }
}
__device__ __forceinline__ M3 mul(const M3 &a, const M3 &b)
{
    M3 c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            double re = a.m[i][0].re * b.m[0][j].re, im = a.m[i][0].re * b.m[0][j].im;
            re = fmx(-a.m[i][0].im, b.m[0][j].im, re);
            im = fmx(a.m[i][0].im, b.m[0][j].re, im);
#pragma unroll
            for (int k = 1; k < 3; k++) {
                re = fmx(a.m[i][k].re, b.m[k][j].re, re);
                re = fmx(-a.m[i][k].im, b.m[k][j].im, re);
                im = fmx(a.m[i][k].re, b.m[k][j].im, im);
                im = fmx(a.m[i][k].im, b.m[k][j].re, im);
            }
            c.m[i][j] = mk(re, im);
        }
    return c;
}
__device__ __forceinline__ M3 dag(const M3 &a)
{
    M3 c;
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) c.m[i][j] = conjx(a.m[j][i]);
    return c;
}
__device__ __forceinline__ void add_scaled(M3 &acc, double s, const M3 &a)
{
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) acc.m[i][j] = acc.m[i][j] + s * a.m[i][j];
}

// host-built table of the Gell-Mann matrices, complex (re, im)
struct Tabs {
    double2 lam[8][3][3];
};

__device__ __forceinline__ Cd tc(const double2 &v) { return mk(v.x, v.y); }

// g_a = Re tr(T_a M) = -1/2 Im tr(lambda_a M), the entries of the Gell-Mann
// matrices written out
__device__ __forceinline__ void project_generators(const M3 &M, double g[8])
{
    g[0] = -0.5 * (M.m[1][0].im + M.m[0][1].im);
    g[1] = -0.5 * (M.m[0][1].re - M.m[1][0].re);
    g[2] = -0.5 * (M.m[0][0].im - M.m[1][1].im);
    g[3] = -0.5 * (M.m[2][0].im + M.m[0][2].im);
    g[4] = -0.5 * (M.m[0][2].re - M.m[2][0].re);
    g[5] = -0.5 * (M.m[2][1].im + M.m[1][2].im);
    g[6] = -0.5 * (M.m[1][2].re - M.m[2][1].re);
    g[7] = -0.28867513459481288225 * (M.m[0][0].im + M.m[1][1].im - 2.0 * M.m[2][2].im);   // 1 / (2 sqrt 3)
}

__device__ __forceinline__ void site_coords(const Geom &g, long s, int x[4])
{
    x[3] = (int)(s % g.L[3]);
    long t = s / g.L[3];
    x[2] = (int)(t % g.L[2]);
    t /= g.L[2];
    x[1] = (int)(t % g.L[1]);
    x[0] = (int)(t / g.L[1]);
}
__device__ __forceinline__ long site_index(const Geom &g, const int x[4])
{
    return x[3] + (long)g.L[3] * (x[2] + (long)g.L[2] * (x[1] + (long)g.L[1] * x[0]));
}
__device__ __forceinline__ void shift(const Geom &g, int y[4], int mu, int d)
{
    int v = y[mu] + d;
    y[mu] = v < 0 ? v + g.L[mu] : (v >= g.L[mu] ? v - g.L[mu] : v);
}
// U_mu(x) from the native FP64 copy ([p][mu][9][Vh] at rank site >> 1)
__device__ __forceinline__ M3 link_at(const Geom &g, const double2 *__restrict__ U, const int x[4], int mu)
{
    const long s = site_index(g, x);
    const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
    const double2 *b = U + (long)((p * 4 + mu) * 9) * g.Vh + (s >> 1);
    M3 u;
#pragma unroll
    for (int e = 0; e < 9; e++) u.m[e / 3][e % 3] = tc(b[e * (long)g.Vh]);
    return u;
}
__device__ __forceinline__ void spinor_at(const double2 *f, long s, Cd v[4][3])
{
#pragma unroll
    for (int sp = 0; sp < 4; sp++)
#pragma unroll
        for (int c = 0; c < 3; c++) v[sp][c] = tc(f[12 * s + 3 * sp + c]);
}

__device__ __forceinline__ void store_grad(double *gout, long l, const double gv[8], double scale, int accumulate)
{
#pragma unroll
    for (int a = 0; a < 8; a++) gout[8 * l + a] = (accumulate ? gout[8 * l + a] : 0.0) + scale * gv[a];
}

// the link of this thread: direction and parity from the block's y index, rank
// from x; false past the last rank
__device__ __forceinline__ bool my_link(const Geom &g, int &mu, int &p, int &r, int x[4], long &l)
{
    mu = blockIdx.y >> 1;
    p = blockIdx.y & 1;
    r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= g.Vh) return false;
    rank_coords(g, p, r, x);
    l = 4 * site_index(g, x) + mu;
    return true;
}

// ------------------------------------------------------------------ hops
// h = psi_up + sgn e_mu psi_lo, the half spinor of (1 + sgn g_mu) psi
__device__ __forceinline__ void half_spinor(int mu, double sgn, const Cd v[4][3], Cd h[2][3])
{
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const Cd l0 = v[2][c], l1 = v[3][c];
        Cd e0, e1;
        switch (mu) {
            case 0: e0 = -l0; e1 = -l1; break;
            case 1: e0 = timesmI(l1); e1 = timesmI(l0); break;
            case 2: e0 = -l1; e1 = l0; break;
            default: e0 = timesmI(l0); e1 = timesI(l1); break;
        }
        h[0][c] = mk(fmx(sgn, e0.re, v[0][c].re), fmx(sgn, e0.im, v[0][c].im));
        h[1][c] = mk(fmx(sgn, e1.re, v[1][c].re), fmx(sgn, e1.im, v[1][c].im));
    }
}
// acc[k][i] += a[k] conj(b[i])
__device__ __forceinline__ void outer_add(M3 &acc, const Cd a[3], const Cd b[3])
{
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
        for (int i = 0; i < 3; i++) {
            Cd &m = acc.m[k][i];
            m.re = fmx(a[k].re, b[i].re, m.re);
            m.re = fmx(a[k].im, b[i].im, m.re);
            m.im = fmx(a[k].im, b[i].re, m.im);
            m.im = fmx(-a[k].re, b[i].im, m.im);
        }
}

// The lower half of (1 -+ g_mu) psi follows from the upper half h, so the spin
// sums of B1 and B2 are sum_{s < 2} h_s(X) h_s(Y)^dag with the same projection
// of both fields, and M = -1/2 s U (B1 + B2^dag).
__global__ void __launch_bounds__(128) k_force_hop(Geom g, const double2 *__restrict__ U, const double2 *__restrict__ X,
                                                   const double2 *__restrict__ Y, double *gout, double scale,
                                                   int accumulate)
{
    int mu, p, r, x[4];
    long l;
    if (!my_link(g, mu, p, r, x, l)) return;
    int y[4] = {x[0], x[1], x[2], x[3]};
    shift(g, y, mu, +1);
    const long s = site_index(g, x), sy = site_index(g, y);
    const double sgn = (mu == 0 && x[0] == g.L[0] - 1) ? double(g.bc_t) : 1.0;
    M3 W = m3_zero();
    Cd v[4][3], a[2][3], b[2][3];
    // B1 = sum_s [(1 - g_mu) X(x+mu)]_s Y(x)_s^dag
    spinor_at(X, sy, v);
    half_spinor(mu, -1.0, v, a);
    spinor_at(Y, s, v);
    half_spinor(mu, -1.0, v, b);
    outer_add(W, a[0], b[0]);
    outer_add(W, a[1], b[1]);
    // B2^dag = sum_s Y(x+mu)_s [(1 + g_mu) X(x)]_s^dag
    spinor_at(Y, sy, v);
    half_spinor(mu, +1.0, v, a);
    spinor_at(X, s, v);
    half_spinor(mu, +1.0, v, b);
    outer_add(W, a[0], b[0]);
    outer_add(W, a[1], b[1]);
    double gv[8];
    project_generators(mul(link_at(g, U, x, mu), W), gv);
    store_grad(gout, l, gv, -0.5 * sgn * scale, accumulate);
}

// ------------------------------------------------------------------ clover
// plane index of (rho, sigma), rho < sigma
__device__ __forceinline__ int plane_of(int r, int s) { return r == 0 ? s - 1 : (r == 1 ? s + 1 : 5); }

// Om[parity][plane][9][Vh].  In the chiral basis sigma is block diagonal, with
// Pauli matrix s_k of the upper / lower block in the planes
//   sigma_0k: +s_k / -s_k,   sigma_23, sigma_12: -s_1, -s_3 / -s_1, -s_3,
//   sigma_13: +s_2 / +s_2,
// so six colour matrices T_k^h = sum_ab (s_k)_ab N_ab (N_ab the colour block of
// M between spins b and a of half h) give all planes: Lam = (i/4)(+-T^0 +-T^1),
// Om = (i/4)(+-G^0 +-G^1) with G = T + T^dag.
// G[k] = T_k + T_k^dag of one half from its N_ab
__device__ __forceinline__ void pauli_sums(const M3 &n00, const M3 &n01, const M3 &n10, const M3 &n11, M3 G[3])
{
#pragma unroll
    for (int k = 0; k < 3; k++)
#pragma unroll
        for (int i = 0; i < 3; i++) {
            // T1 = N01 + N10, T2 = -i N01 + i N10, T3 = N00 - N11
            const Cd t1 = n01.m[k][i] + n10.m[k][i], t1t = n01.m[i][k] + n10.m[i][k];
            const Cd t2 = timesI(n10.m[k][i] - n01.m[k][i]), t2t = timesI(n10.m[i][k] - n01.m[i][k]);
            const Cd t3 = n00.m[k][i] - n11.m[k][i], t3t = n00.m[i][k] - n11.m[i][k];
            G[0].m[k][i] = t1 + conjx(t1t);
            G[1].m[k][i] = t2 + conjx(t2t);
            G[2].m[k][i] = t3 + conjx(t3t);
        }
}

// src = 0: M = X Y^dag on every site; src = 1: M = A^-1 on the sites of parity
// par (blockIdx.y runs over the parities written)
__global__ void __launch_bounds__(128) k_omega(Geom g, int src, const double2 *__restrict__ X,
                                               const double2 *__restrict__ Y, const double2 *__restrict__ Ai,
                                               int par, double2 *Om)
{
    const int p = src == 0 ? (int)blockIdx.y : par;
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= g.Vh) return;
    const long Vh = g.Vh;
    M3 G[2][3];
    if (src == 0) {
        int x[4];
        rank_coords(g, p, r, x);
        const long s = site_index(g, x);
        Cd Xs[4][3], Ys[4][3];
        spinor_at(X, s, Xs);
        spinor_at(Y, s, Ys);
#pragma unroll
        for (int h = 0; h < 2; h++) {
            M3 n[2][2];
#pragma unroll
            for (int a = 0; a < 2; a++)
#pragma unroll
                for (int b = 0; b < 2; b++) {
                    n[a][b] = m3_zero();
                    outer_add(n[a][b], Xs[2 * h + b], Ys[2 * h + a]);
                }
            pauli_sums(n[0][0], n[0][1], n[1][0], n[1][1], G[h]);
        }
    } else {
#pragma unroll
        for (int h = 0; h < 2; h++) {   // packed Hermitian block: 6 real diagonal, 15 upper entries
            const double2 *bp = Ai + (long)(18 * h) * Vh + r;
            double d[6];
            Cd blk[6][6];
#pragma unroll
            for (int q = 0; q < 3; q++) {
                const double2 v = bp[q * Vh];
                d[2 * q] = v.x;
                d[2 * q + 1] = v.y;
            }
            int kk = 0;
#pragma unroll
            for (int i = 0; i < 6; i++) {
                blk[i][i] = mk(d[i], 0.0);
#pragma unroll
                for (int j = i + 1; j < 6; j++) {
                    const Cd o = tc(bp[(3 + kk++) * Vh]);
                    blk[i][j] = o;
                    blk[j][i] = conjx(o);
                }
            }
            M3 n[2][2];
#pragma unroll
            for (int a = 0; a < 2; a++)
#pragma unroll
                for (int b = 0; b < 2; b++)
#pragma unroll
                    for (int k = 0; k < 3; k++)
#pragma unroll
                        for (int i = 0; i < 3; i++) n[a][b].m[k][i] = blk[3 * b + k][3 * a + i];
            pauli_sums(n[0][0], n[0][1], n[1][0], n[1][1], G[h]);
        }
    }
    double2 *op = Om + (long)p * 54 * Vh + r;
    auto put = [&](int pl, int e, Cd t) {   // (i/4) t
        op[(pl * 9L + e) * Vh] = make_double2(-0.25 * t.im, 0.25 * t.re);
    };
#pragma unroll
    for (int e = 0; e < 9; e++) {
        const int k = e / 3, i = e % 3;
        const Cd u0 = G[0][0].m[k][i], l0 = G[1][0].m[k][i], u1 = G[0][1].m[k][i], l1 = G[1][1].m[k][i],
                 u2 = G[0][2].m[k][i], l2 = G[1][2].m[k][i];
        put(0, e, u0 - l0);      // 01
        put(1, e, u1 - l1);      // 02
        put(2, e, u2 - l2);      // 03
        put(3, e, -(u2 + l2));   // 12
        put(4, e, u1 + l1);      // 13
        put(5, e, -(u0 + l0));   // 23
    }
}

__device__ __forceinline__ M3 om_at(const Geom &g, const double2 *__restrict__ Om, const int x[4], int pl)
{
    const int p = (x[0] + x[1] + x[2] + x[3]) & 1;
    const double2 *b = Om + (long)(p * 54 + pl * 9) * g.Vh + coords_rank(g, x);
    M3 m;
#pragma unroll
    for (int e = 0; e < 9; e++) m.m[e / 3][e % 3] = tc(b[e * (long)g.Vh]);
    return m;
}

// The places where U_mu(x) sits in a clover leaf, summed.  The leaf of plane
// (nu, mu) is the adjoint of that of (mu, nu) and Om changes sign with the
// order, so the two orders contribute equally and one is taken, twice.  With
// the staples a b c = U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag and
// a' b' c' = U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu), D = a b c - a' b' c'
// and Om at the four corners of each staple, the eight leaves of a plane give
//   W = Om(x+mu) D + D Om(x) + (a Om(x+mu+nu) b + a b Om(x+nu)) c
//                            - (a' Om(x+mu-nu) b' + a' b' Om(x-nu)) c',
// M = (c_sw / 4) U sum_nu (+-) W: 14 products a plane and 43 a link where the
// sum over (order, leaf, place) took 288.  Om is nonzero on one parity only in
// the log det force: SEL = 1 (the parity of x) and SEL = 2 (the other one) leave
// out the products with zero.  Measured at 32 x 16^3: 52.7 -> 4.29 ms (SEL = 0;
// floor of the FP64 pipe 3.9), log det 52.7 -> 1.80 + 1.51 ms.
template <int SEL>
__global__ void __launch_bounds__(64) k_force_clover(Geom g, const double2 *__restrict__ U,
                                                     const double2 *__restrict__ Om, double coef, double *gout,
                                                     double scale, int accumulate, int par)
{
    constexpr bool AT_X = SEL != 2, AT_N = SEL != 1;   // Om nonzero at x, x+mu+-nu / at x+mu, x+-nu
    const int mu = SEL == 0 ? blockIdx.y >> 1 : blockIdx.y;
    const int p = SEL == 0 ? (int)(blockIdx.y & 1) : (SEL == 1 ? par : 1 - par);
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= g.Vh) return;
    int x[4];
    rank_coords(g, p, r, x);
    const long l = 4 * site_index(g, x) + mu;
    M3 W = m3_zero();
#pragma unroll 1
    for (int k = 1; k < 4; k++) {
        const int nu = (mu + k) & 3;
        const int pl = plane_of(min(mu, nu), max(mu, nu));
        int xm[4] = {x[0], x[1], x[2], x[3]};
        shift(g, xm, mu, +1);
        M3 Wn = m3_zero(), D;
#pragma unroll 1
        for (int dn = 0; dn < 2; dn++) {   // the staple at +nu, then the one at -nu
            int ys[4] = {x[0], x[1], x[2], x[3]}, yn[4] = {x[0], x[1], x[2], x[3]}, xmn[4] = {xm[0], xm[1], xm[2], xm[3]};
            shift(g, yn, nu, dn ? -1 : +1);    // the staple's mu link starts here
            shift(g, xmn, nu, dn ? -1 : +1);   // and ends here
            M3 a = link_at(g, U, dn ? xmn : xm, nu);
            M3 c = link_at(g, U, dn ? yn : ys, nu);
            if (dn)
                a = dag(a);
            else
                c = dag(c);
            const M3 b = dag(link_at(g, U, yn, mu));
            const M3 ab = mul(a, b);
            const M3 S = mul(ab, c);
            M3 t;
            if (AT_X) {
                t = mul(mul(a, om_at(g, Om, xmn, pl)), b);
                if (AT_N) mul_add(t, ab, om_at(g, Om, yn, pl));
            } else {
                t = mul(ab, om_at(g, Om, yn, pl));
            }
            if (dn == 0) {
                D = S;
                mul_add(Wn, t, c);
            } else {
                add_scaled(D, -1.0, S);
                add_scaled(Wn, -1.0, mul(t, c));
            }
        }
        if (AT_X) mul_add(Wn, D, om_at(g, Om, x, pl));
        if (AT_N) mul_add(Wn, om_at(g, Om, xm, pl), D);
        add_scaled(W, mu < nu ? 1.0 : -1.0, Wn);   // Om_{nu mu} = -Om_{mu nu}
    }
    double gv[8];
    project_generators(mul(link_at(g, U, x, mu), W), gv);
    store_grad(gout, l, gv, 0.25 * coef * scale, accumulate);
}

// ------------------------------------------------------------------ gauge
__global__ void __launch_bounds__(128) k_force_gauge(Geom g, const double2 *__restrict__ U, double beta, double *gout,
                                                     double scale, int accumulate)
{
    int mu, p, r, x[4];
    long l;
    if (!my_link(g, mu, p, r, x, l)) return;
    M3 st = m3_zero();
#pragma unroll 1
    for (int k = 1; k < 4; k++) {
        const int nu = (mu + k) & 3;
        int xm[4] = {x[0], x[1], x[2], x[3]}, xn[4] = {x[0], x[1], x[2], x[3]};
        shift(g, xm, mu, +1);
        shift(g, xn, nu, +1);
        // up: U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
        mul_add(st, mul(link_at(g, U, xm, nu), dag(link_at(g, U, xn, mu))), dag(link_at(g, U, x, nu)));
        // down: U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu)
        int xmn[4] = {xm[0], xm[1], xm[2], xm[3]}, xd[4] = {x[0], x[1], x[2], x[3]};
        shift(g, xmn, nu, -1);
        shift(g, xd, nu, -1);
        mul_add(st, mul(dag(link_at(g, U, xmn, nu)), dag(link_at(g, U, xd, mu))), link_at(g, U, xd, nu));
    }
    double gv[8];
    project_generators(mul(link_at(g, U, x, mu), st), gv);
    store_grad(gout, l, gv, -beta / 3.0 * scale, accumulate);
}

// per-site sum over the six planes of 1 - Re tr U_P / 3
__global__ void __launch_bounds__(128) k_plaq_site(Geom g, const double2 *__restrict__ U, double *out)
{
    const long s = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (s >= g.V) return;
    int x[4];
    site_coords(g, s, x);
    double acc = 0;
    for (int mu = 0; mu < 4; mu++)
        for (int nu = mu + 1; nu < 4; nu++) {
            int xm[4] = {x[0], x[1], x[2], x[3]}, xn[4] = {x[0], x[1], x[2], x[3]};
            shift(g, xm, mu, +1);
            shift(g, xn, nu, +1);
            const M3 P = mul(mul(link_at(g, U, x, mu), link_at(g, U, xm, nu)),
                             mul(dag(link_at(g, U, xn, mu)), dag(link_at(g, U, x, nu))));
            acc += 1.0 - (P.m[0][0].re + P.m[1][1].re + P.m[2][2].re) / 3.0;
        }
    out[s] = acc;
}

// fixed-order sum of n doubles (one CTA, deterministic)
__global__ void k_sum_md(const double *x, long n, double *out)
{
    __shared__ double sh[256];
    double s = 0;
    for (long i = threadIdx.x; i < n; i += blockDim.x) s += x[i];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0) *out = sh[0];
}

// ------------------------------------------------------------------ MD step
// U <- exp(dt P) U on canonical links [site][mu][3][3] (complex), P = sum_a p^a T_a
__global__ void __launch_bounds__(128) k_move_links(long nlink, const double *__restrict__ p, double dt, double2 *U,
                                                    Tabs T)
{
    const long l = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (l >= nlink) return;
    M3 P = m3_zero();
    for (int a = 0; a < 8; a++) {
        const double c = dt * p[8 * l + a];
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) P.m[i][j] = P.m[i][j] + (0.5 * c) * timesI(tc(T.lam[a][i][j]));
    }
    // scaling: |P| / 2^k <= 1/2 in the max-row-sum norm
    double nrm = 0;
    for (int i = 0; i < 3; i++) {
        double r = 0;
        for (int j = 0; j < 3; j++) r += sqrt(P.m[i][j].re * P.m[i][j].re + P.m[i][j].im * P.m[i][j].im);
        nrm = fmax(nrm, r);
    }
    int k = 0;
    while (nrm > 0.5 && k < 60) {
        nrm *= 0.5;
        k++;
    }
    const double sc = ldexp(1.0, -k);
    M3 A;
    for (int i = 0; i < 3; i++)
        for (int j = 0; j < 3; j++) A.m[i][j] = sc * P.m[i][j];
    // Taylor series to order 20: remainder below 0.5^21 / 21! relative
    M3 E = m3_one(), term = m3_one();
    for (int n = 1; n <= 20; n++) {
        term = mul(term, A);
        for (int i = 0; i < 3; i++)
            for (int j = 0; j < 3; j++) term.m[i][j] = (1.0 / n) * term.m[i][j];
        add_scaled(E, 1.0, term);
    }
    for (int q = 0; q < k; q++) E = mul(E, E);
    M3 u;
    double2 *up = U + 9 * l;
    for (int e = 0; e < 9; e++) u.m[e / 3][e % 3] = tc(up[e]);
    const M3 v = mul(E, u);
    for (int e = 0; e < 9; e++) up[e] = make_double2(v.m[e / 3][e % 3].re, v.m[e / 3][e % 3].im);
}

__global__ void k_axpy_real(long n, double a, const double *__restrict__ x, double *y)
{
    for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < n; i += (long)gridDim.x * blockDim.x)
        y[i] += a * x[i];
}

// ------------------------------------------------------------------ host
Tabs make_tabs()
{
    Tabs T{};
    auto set = [](double2 &d, double re, double im) { d = make_double2(re, im); };
    // Gell-Mann matrices
    const double r3 = 1.0 / std::sqrt(3.0);
    set(T.lam[0][0][1], 1, 0);
    set(T.lam[0][1][0], 1, 0);
    set(T.lam[1][0][1], 0, -1);
    set(T.lam[1][1][0], 0, 1);
    set(T.lam[2][0][0], 1, 0);
    set(T.lam[2][1][1], -1, 0);
    set(T.lam[3][0][2], 1, 0);
    set(T.lam[3][2][0], 1, 0);
    set(T.lam[4][0][2], 0, -1);
    set(T.lam[4][2][0], 0, 1);
    set(T.lam[5][1][2], 1, 0);
    set(T.lam[5][2][1], 1, 0);
    set(T.lam[6][1][2], 0, -1);
    set(T.lam[6][2][1], 0, 1);
    set(T.lam[7][0][0], r3, 0);
    set(T.lam[7][1][1], r3, 0);
    set(T.lam[7][2][2], -2 * r3, 0);
    return T;
}

const Tabs &tabs()
{
    static const Tabs T = make_tabs();
    return T;
}

// one block row per (direction, parity)
dim3 grid_links(const lqcd_ctx *c, int tpb, int rows = 8) { return dim3(div_up(c->g.Vh, tpb), rows); }

lqcd_status need_state(lqcd_ctx *c)
{
    if (!c->have_gauge) return set_err(c, LQCD_ERR_STATE, "gauge field not set");
    if (!c->have_clover) return set_err(c, LQCD_ERR_STATE, "clover term not built");
    return LQCD_OK;
}

// g (+)= scale * Re <Y, dD X> (X, Y canonical full FP64 fields on the device)
lqcd_status force_dD(lqcd_ctx *c, const double *X, const double *Y, double *g, double scale, int accumulate)
{
    LQCD_TRY(need_state(c));
    k_force_hop<<<grid_links(c, 128), 128, 0, c->stream>>>(c->g, c->U64, (const double2 *)X, (const double2 *)Y, g,
                                                           scale, accumulate);
    c->n_kernel_launches++;
    LQCD_LAUNCH_CHECK(c);
    if (c->csw != 0.0) {
        void *om;
        LQCD_TRY(ws_get(c, WS_MD_OMEGA, (size_t)c->g.V * 6 * 9 * sizeof(double2), &om));
        k_omega<<<grid_links(c, 128, 2), 128, 0, c->stream>>>(c->g, 0, (const double2 *)X, (const double2 *)Y, nullptr,
                                                              0, (double2 *)om);
        c->n_kernel_launches++;
        LQCD_LAUNCH_CHECK(c);
        k_force_clover<0><<<grid_links(c, 64), 64, 0, c->stream>>>(c->g, c->U64, (const double2 *)om, c->csw, g, scale,
                                                                   1, 0);
        c->n_kernel_launches++;
        LQCD_LAUNCH_CHECK(c);
    }
    return LQCD_OK;
}

// g (+)= scale * d log|det A_parity| / d eps = scale * sum_y Re tr(A^-1 dA)
lqcd_status force_logdet(lqcd_ctx *c, int parity, double *g, double scale, int accumulate)
{
    LQCD_TRY(need_state(c));
    if (c->csw == 0.0) {   // A = (4 + m0) 1 does not depend on the links
        if (!accumulate) LQCD_TRY(blas_zero(c, (size_t)c->g.V * 32 * sizeof(double), g));
        return LQCD_OK;
    }
    void *om;
    LQCD_TRY(ws_get(c, WS_MD_OMEGA, (size_t)c->g.V * 6 * 9 * sizeof(double2), &om));
    k_omega<<<grid_links(c, 128, 1), 128, 0, c->stream>>>(c->g, 1, nullptr, nullptr, c->Ai64[parity], parity,
                                                          (double2 *)om);
    c->n_kernel_launches++;
    LQCD_LAUNCH_CHECK(c);
    k_force_clover<1><<<grid_links(c, 64, 4), 64, 0, c->stream>>>(c->g, c->U64, (const double2 *)om, c->csw, g, scale,
                                                                  accumulate, parity);
    k_force_clover<2><<<grid_links(c, 64, 4), 64, 0, c->stream>>>(c->g, c->U64, (const double2 *)om, c->csw, g, scale,
                                                                  accumulate, parity);
    c->n_kernel_launches += 2;
    LQCD_LAUNCH_CHECK(c);
    return LQCD_OK;
}

lqcd_status force_gauge(lqcd_ctx *c, double beta, double *g, double scale, int accumulate)
{
    if (!c->have_gauge) return set_err(c, LQCD_ERR_STATE, "gauge field not set");
    k_force_gauge<<<grid_links(c, 128), 128, 0, c->stream>>>(c->g, c->U64, beta, g, scale, accumulate);
    c->n_kernel_launches++;
    LQCD_LAUNCH_CHECK(c);
    return LQCD_OK;
}

lqcd_status gauge_action(lqcd_ctx *c, double beta, double *S)
{
    if (!c->have_gauge) return set_err(c, LQCD_ERR_STATE, "gauge field not set");
    void *w;
    LQCD_TRY(ws_get(c, WS_MD_SCRATCH, (size_t)c->g.V * sizeof(double) + 64, &w));
    double *site = (double *)w;
    k_plaq_site<<<div_up(c->g.V, 128), 128, 0, c->stream>>>(c->g, c->U64, site);
    c->n_kernel_launches++;
    LQCD_LAUNCH_CHECK(c);
    k_sum_md<<<1, 256, 0, c->stream>>>(site, c->g.V, c->red_out);
    c->n_kernel_launches++;
    LQCD_LAUNCH_CHECK(c);
    double h = 0;
    LQCD_CUDA_CHECK(c, cudaMemcpyAsync(&h, c->red_out, sizeof(double), cudaMemcpyDeviceToHost, c->stream));
    LQCD_CUDA_CHECK(c, cudaStreamSynchronize(c->stream));
    *S = beta * h;
    return LQCD_OK;
}

// The pseudofermion field of S_pf = |Dhat^-1 phi|^2 and its gradient
// -2 Re <Y, dD X>, X = (x_e, -A_oo^-1 H_oe x_e), Y = (y_e, -A_oo^-1 H_eo^dag y_e),
// x_e = Dhat^-1 phi, y_e = Dhat^-dag x_e = gamma5 Dhat^-1 gamma5 x_e; with these
// completions <Y, dD X> = <y_e, dDhat x_e>.  S (optional) = |x_e|^2.
lqcd_status force_pf(lqcd_ctx *c, const lqcd_solver_params *sp, const double *phi_e, double *g, double scale,
                     int accumulate, double *S, lqcd_solve_info *info)
{
    LQCD_TRY(need_state(c));
    const long Vh = c->g.Vh;
    const size_t hb = native_half_bytes(c, LQCD_F64);   // one native half field
    const long ne = 24 * Vh;                              // doubles in an even canonical field
    void *w;
    // canonical: x_e, t_e, y_e (even), X, Y (full); native: three full fields
    LQCD_TRY(ws_get(c, WS_MD_FIELDS, 3 * ne * sizeof(double) + 2 * 2 * ne * sizeof(double) + 6 * hb, &w));
    double *xe = (double *)w, *te = xe + ne, *ye = te + ne, *Xf = ye + ne, *Yf = Xf + 2 * ne;
    double2 *nx = (double2 *)(Yf + 2 * ne), *ny = nx + 24 * Vh, *nt = ny + 24 * Vh;
    lqcd_solve_info inf[2];
    LQCD_TRY(lqcd_solve_dhat(c, sp, phi_e, xe, 1, &inf[0]));
    // gamma5 on a canonical even field: spins 2, 3 change sign
    auto g5 = [&](const double *in, double *out) -> lqcd_status {
        LQCD_TRY(pack_field(c, LQCD_F64, 1, in, nx, 1, false));
        LQCD_TRY(blas_gamma5_native64(c, 1, nx, nx));
        return pack_field(c, LQCD_F64, 1, out, nx, 1, true);
    };
    LQCD_TRY(g5(xe, te));
    LQCD_TRY(lqcd_solve_dhat(c, sp, te, ye, 1, &inf[1]));
    LQCD_TRY(g5(ye, ye));
    if (info) {
        info[0] = inf[0];
        info[1] = inf[1];
    }
    // X = (x_e, -A_oo^-1 H_oe x_e) in native order [even][odd]
    const long hh = 12 * Vh;
    LQCD_TRY(pack_field(c, LQCD_F64, 1, xe, nx, 1, false));
    LQCD_TRY(dirac_hop_parity(c, LQCD_F64, 1, nx, nt, hh, hh, 1));
    LQCD_TRY(clover_apply_native64(c, 1, 1, nt, nx + hh));
    LQCD_TRY(blas_scal(c, 2 * hh, -1.0, 0.0, (double *)(nx + hh)));
    // Y = (y_e, -A_oo^-1 gamma5 H_oe gamma5 y_e)
    LQCD_TRY(pack_field(c, LQCD_F64, 1, ye, ny, 1, false));
    LQCD_TRY(blas_gamma5_native64(c, 1, ny, nt));
    LQCD_TRY(dirac_hop_parity(c, LQCD_F64, 1, nt, nt + hh, hh, hh, 1));
    LQCD_TRY(blas_gamma5_native64(c, 1, nt + hh, nt));
    LQCD_TRY(clover_apply_native64(c, 1, 1, nt, ny + hh));
    LQCD_TRY(blas_scal(c, 2 * hh, -1.0, 0.0, (double *)(ny + hh)));
    LQCD_TRY(pack_field(c, LQCD_F64, 2, Xf, nx, 1, true));
    LQCD_TRY(pack_field(c, LQCD_F64, 2, Yf, ny, 1, true));
    LQCD_TRY(force_dD(c, Xf, Yf, g, -2.0 * scale, accumulate));
    if (S) {
        double n2 = 0;
        LQCD_TRY(blas_norm2(c, ne, xe, &n2));
        *S = n2;
    }
    lqcd_status st = inf[0].status != LQCD_OK ? inf[0].status : inf[1].status;
    if (st != LQCD_OK) return set_err(c, st, "pseudofermion force: solve did not converge");
    return LQCD_OK;
}

// total gradient of S = S_g + |Dhat^-1 phi|^2 - 2 log|det A_oo|
lqcd_status md_gradient(lqcd_ctx *c, const lqcd_md_params *mp, const double *phi_e, double *g, double *S,
                        lqcd_solve_info *info)
{
    LQCD_TRY(force_gauge(c, mp->beta, g, 1.0, 0));
    double spf = 0;
    LQCD_TRY(force_pf(c, &mp->solver, phi_e, g, 1.0, 1, S ? &spf : nullptr, info));
    LQCD_TRY(force_logdet(c, 1, g, -2.0, 1));
    if (S) {
        double sg;
        LQCD_TRY(gauge_action(c, mp->beta, &sg));
        *S = sg + spf - 2.0 * c->logdet_o;
    }
    return LQCD_OK;
}

lqcd_status check_md(lqcd_ctx *c, const lqcd_md_params *mp)
{
    if (!mp) return set_err(c, LQCD_ERR_ARG, "null MD parameters");
    if (mp->nsteps < 0 || !(std::isfinite(mp->dt)) || !(std::isfinite(mp->beta)))
        return set_err(c, LQCD_ERR_ARG, "bad MD parameters");
    return LQCD_OK;
}

}  // namespace

extern "C" {

lqcd_status lqcd_force_dD(lqcd_ctx *c, const double *X, const double *Y, double *g)
{
    if (!c || !X || !Y || !g) return set_err(c, LQCD_ERR_ARG, "null argument");
    return force_dD(c, X, Y, g, 1.0, 0);
}

lqcd_status lqcd_force_logdet(lqcd_ctx *c, int parity, double *g)
{
    if (!c || !g || parity < 0 || parity > 1) return set_err(c, LQCD_ERR_ARG, "bad argument");
    return force_logdet(c, parity, g, 1.0, 0);
}

lqcd_status lqcd_gauge_action(lqcd_ctx *c, double beta, double *S)
{
    if (!c || !S) return set_err(c, LQCD_ERR_ARG, "null argument");
    return gauge_action(c, beta, S);
}

lqcd_status lqcd_force_gauge(lqcd_ctx *c, double beta, double *g)
{
    if (!c || !g) return set_err(c, LQCD_ERR_ARG, "null argument");
    return force_gauge(c, beta, g, 1.0, 0);
}

lqcd_status lqcd_force_pf(lqcd_ctx *c, const lqcd_solver_params *sp, const double *phi_e, double *g,
                          lqcd_solve_info *info)
{
    if (!c || !sp || !phi_e || !g) return set_err(c, LQCD_ERR_ARG, "null argument");
    return force_pf(c, sp, phi_e, g, 1.0, 0, nullptr, info);
}

lqcd_status lqcd_md_gradient(lqcd_ctx *c, const lqcd_md_params *mp, const double *phi_e, double *g, double *S)
{
    if (!c || !phi_e || !g) return set_err(c, LQCD_ERR_ARG, "null argument");
    LQCD_TRY(check_md(c, mp));
    LQCD_TRY(need_state(c));
    return md_gradient(c, mp, phi_e, g, S, nullptr);
}

lqcd_status lqcd_md_leapfrog(lqcd_ctx *c, const lqcd_md_params *mp, double *U, double *p, const double *phi_e)
{
    if (!c || !U || !p || !phi_e) return set_err(c, LQCD_ERR_ARG, "null argument");
    LQCD_TRY(check_md(c, mp));
    LQCD_TRY(need_state(c));
    const double kappa = c->kappa, csw = c->csw;
    const long nl = 4L * c->g.V, np = 8 * nl;
    void *w;
    LQCD_TRY(ws_get(c, WS_MD_GRAD, np * sizeof(double), &w));
    double *g = (double *)w;
    const int gr = (int)std::min<long>(4 * 152, div_up(np, 256));
    // the field in U is the one the context holds: its gradient starts the step
    LQCD_TRY(md_gradient(c, mp, phi_e, g, nullptr, nullptr));
    for (int step = 0; step < mp->nsteps; step++) {
        k_axpy_real<<<gr, 256, 0, c->stream>>>(np, -0.5 * mp->dt, g, p);
        c->n_kernel_launches++;
        LQCD_LAUNCH_CHECK(c);
        k_move_links<<<div_up(nl, 128), 128, 0, c->stream>>>(nl, p, mp->dt, (double2 *)U, tabs());
        c->n_kernel_launches++;
        LQCD_LAUNCH_CHECK(c);
        LQCD_TRY(lqcd_set_gauge(c, U));
        LQCD_TRY(clover_build(c, kappa, csw, nullptr, nullptr));
        LQCD_TRY(md_gradient(c, mp, phi_e, g, nullptr, nullptr));
        k_axpy_real<<<gr, 256, 0, c->stream>>>(np, -0.5 * mp->dt, g, p);
        c->n_kernel_launches++;
        LQCD_LAUNCH_CHECK(c);
    }
    LQCD_CUDA_CHECK(c, cudaStreamSynchronize(c->stream));
    return LQCD_OK;
}

}  // extern "C"
