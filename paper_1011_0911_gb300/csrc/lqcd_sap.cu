// Schwarz alternating procedure (the Schwarz preconditioner of the GCR solver
// named in Sec. 3-4).  The lattice is tiled by bs0 x bs1 x bs2 x bs3 blocks,
// coloured by the parity of their block coordinates.  One sweep over a colour
// solves D_blk chi = r on every block of that colour approximately and adds
// chi to psi; the residual r = eta - D psi is then recomputed.
//
// Block solve (one CTA per block, all block vectors in shared memory):
//   b_e = r_e - H_eo,blk A_oo^-1 r_o
//   nmr MinRes steps on Dhat_blk = A_ee - H_eo,blk A_oo^-1 H_oe,blk from 0:
//       p = Dhat_blk rho, alpha = <p,rho>/<p,p>, chi_e += alpha rho, rho -= alpha p
//   chi_o = A_oo^-1 (r_o - H_oe,blk chi_e)
// H_blk keeps only hops whose both ends lie in the block (Dirichlet); a block
// that spans a whole lattice direction keeps the wrapped hop of that direction.
#include <algorithm>
#include <list>
#include <type_traits>
#include <vector>

#include "lqcd_f16s.cuh"
#include "lqcd_internal.cuh"
#include "lqcd_stencil.cuh"
#include "lqcd_tune.h"

namespace {

struct BlkGeom {
    int bs[4];
    int nb[4];
    int nh;          // sites of one parity per block
    int bs3h;
    int wrap[4];     // block spans the whole direction
};

// storage per precision tag: arithmetic type, spinor unit, link and clover
// element types, and the length of one native half field in spinor units
template <int P>
struct SapT;
template <>
struct SapT<LQCD_F64> {
    using R = double;
    using SP = double2;
    using LK = double2;
    using CL = double2;
    static __host__ __device__ long half(long Vh) { return 12 * Vh; }
};
template <>
struct SapT<LQCD_F32> {
    using R = float;
    using SP = float4;
    using LK = float4;
    using CL = float4;
    static __host__ __device__ long half(long Vh) { return 6 * Vh; }
};
template <>
struct SapT<LQCD_F16S> {
    using R = float;
    using SP = h16s;
    using LK = uint2;
    using CL = uint2;
    static __host__ __device__ long half(long Vh) { return f16s_half_units(Vh); }
};

// global native accessors (duplicated minimal forms of the stencil loaders)
__device__ __forceinline__ void gload(const double2 *f, long Vh, long r, cx<double> v[12])
{
#pragma unroll
    for (int c = 0; c < 12; c++) {
        double2 t = f[c * Vh + r];
        v[c] = mk(t.x, t.y);
    }
}
__device__ __forceinline__ void gload(const float4 *f, long Vh, long r, cx<float> v[12])
{
#pragma unroll
    for (int q = 0; q < 6; q++) {
        float4 t = f[q * Vh + r];
        v[2 * q] = mk(t.x, t.y);
        v[2 * q + 1] = mk(t.z, t.w);
    }
}
__device__ __forceinline__ void gadd(double2 *f, long Vh, long r, const cx<double> v[12])
{
#pragma unroll
    for (int c = 0; c < 12; c++) {
        double2 t = f[c * Vh + r];
        f[c * Vh + r] = make_double2(t.x + v[c].re, t.y + v[c].im);
    }
}
__device__ __forceinline__ void gadd(float4 *f, long Vh, long r, const cx<float> v[12])
{
#pragma unroll
    for (int q = 0; q < 6; q++) {
        float4 t = f[q * Vh + r];
        f[q * Vh + r] = make_float4(t.x + v[2 * q].re, t.y + v[2 * q].im, t.z + v[2 * q + 1].re,
                                    t.w + v[2 * q + 1].im);
    }
}
__device__ __forceinline__ void glink(const double2 *U, long Vh, int p, int mu, long r, cx<double> u[3][3])
{
    const double2 *b = U + (long)((p * 4 + mu) * 9) * Vh + r;
#pragma unroll
    for (int e = 0; e < 9; e++) {
        double2 t = __ldg(b + e * Vh);
        u[e / 3][e % 3] = mk(t.x, t.y);
    }
}
__device__ __forceinline__ void glink(const float4 *U, long Vh, int p, int mu, long r, cx<float> u[3][3])
{
    const float4 *b = U + (long)((p * 4 + mu) * 3) * Vh + r;
#pragma unroll
    for (int q = 0; q < 3; q++) {
        float4 t = __ldg(b + q * Vh);
        u[(2 * q) / 3][(2 * q) % 3] = mk(t.x, t.y);
        u[(2 * q + 1) / 3][(2 * q + 1) % 3] = mk(t.z, t.w);
    }
    su3_third_row(u);
}
__device__ __forceinline__ void gload(const h16s *f, long Vh, long r, cx<float> v[12]) { f16s_load<false>(f, Vh, r, v); }
__device__ __forceinline__ void gadd(h16s *f, long Vh, long r, const cx<float> v[12])
{
    cx<float> t[12];
    f16s_load<false>(f, Vh, r, t);
#pragma unroll
    for (int c = 0; c < 12; c++) t[c] = t[c] + v[c];
    f16s_store(f, Vh, r, t);
}
__device__ __forceinline__ void glink(const uint2 *U, long Vh, int p, int mu, long r, cx<float> u[3][3])
{
    f16s_link(U, Vh, p, mu, r, u);
}
__device__ __forceinline__ void gclov(const uint2 *A, long Vh, long r, int blk, float d[6], cx<float> o[15])
{
    float v[36];
    f16s_clover(A, Vh, r, blk, v);
#pragma unroll
    for (int i = 0; i < 6; i++) d[i] = v[i];
#pragma unroll
    for (int i = 0; i < 15; i++) o[i] = mk(v[6 + 2 * i], v[7 + 2 * i]);
}
__device__ __forceinline__ void gclov(const double2 *A, long Vh, long r, int blk, double d[6], cx<double> o[15])
{
    const double2 *b = A + (long)(18 * blk) * Vh + r;
#pragma unroll
    for (int i = 0; i < 3; i++) {
        double2 t = __ldg(b + i * Vh);
        d[2 * i] = t.x;
        d[2 * i + 1] = t.y;
    }
#pragma unroll
    for (int i = 0; i < 15; i++) {
        double2 t = __ldg(b + (3 + i) * Vh);
        o[i] = mk(t.x, t.y);
    }
}
__device__ __forceinline__ void gclov(const float4 *A, long Vh, long r, int blk, float d[6], cx<float> o[15])
{
    const float4 *b = A + (long)(9 * blk) * Vh + r;
    float v[36];
#pragma unroll
    for (int q = 0; q < 9; q++) {
        float4 t = __ldg(b + q * Vh);
        v[4 * q] = t.x;
        v[4 * q + 1] = t.y;
        v[4 * q + 2] = t.z;
        v[4 * q + 3] = t.w;
    }
#pragma unroll
    for (int i = 0; i < 6; i++) d[i] = v[i];
#pragma unroll
    for (int i = 0; i < 15; i++) o[i] = mk(v[6 + 2 * i], v[7 + 2 * i]);
}

// w = H v for a packed Hermitian 6x6 block (diagonal d, upper entries o),
// every product entering its sum through a fused multiply-add
template <class R>
__device__ __forceinline__ void herm6_apply(const R d[6], const cx<R> o[15], const cx<R> v[6], cx<R> w[6])
{
    stencil::Herm6<R> h;
#pragma unroll
    for (int i = 0; i < 6; i++) h.d[i] = d[i];
#pragma unroll
    for (int i = 0; i < 15; i++) h.o[i] = o[i];
    stencil::herm_apply(h, v, w);
}

template <class R, class CL>
__device__ __forceinline__ void clov_apply(const CL *A, long Vh, long r, const cx<R> in[12], cx<R> out[12])
{
#pragma unroll
    for (int blk = 0; blk < 2; blk++) {
        R d[6];
        cx<R> o[15];
        gclov(A, Vh, r, blk, d, o);
        herm6_apply(d, o, in + 6 * blk, out + 6 * blk);
    }
}

// shared-memory block field: component-major [12][nh] complex
template <class R>
__device__ __forceinline__ void sload(const cx<R> *s, int nh, int t, cx<R> v[12])
{
#pragma unroll
    for (int c = 0; c < 12; c++) v[c] = s[c * nh + t];
}
template <class R>
__device__ __forceinline__ void sstore(cx<R> *s, int nh, int t, const cx<R> v[12])
{
#pragma unroll
    for (int c = 0; c < 12; c++) s[c * nh + t] = v[c];
}

// projected hop term of direction mu and sense d from the block-local field
// src (opposite parity), accumulated into acc (before the -1/2 factor).
// v = psi[spin][colour] as v[3*spin + colour].
template <class R>
__device__ __forceinline__ void proj_apply(int mu, int sgn, const cx<R> psi[12], const cx<R> u[3][3], bool dag,
                                           R sign, cx<R> acc[12])
{
    cx<R> h[2][3], w[2][3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        cx<R> u0 = psi[c], u1 = psi[3 + c], l0 = psi[6 + c], l1 = psi[9 + c];
        cx<R> el0, el1;  // e_mu l
        switch (mu) {
            case 0: el0 = -l0; el1 = -l1; break;
            case 1: el0 = timesmI(l1); el1 = timesmI(l0); break;
            case 2: el0 = -l1; el1 = l0; break;
            default: el0 = timesmI(l0); el1 = timesI(l1); break;
        }
        if (sgn < 0) {
            h[0][c] = u0 - el0;
            h[1][c] = u1 - el1;
        } else {
            h[0][c] = u0 + el0;
            h[1][c] = u1 + el1;
        }
    }
#pragma unroll
    for (int s = 0; s < 2; s++) {
        if (!dag)
            stencil::su3_vec(u, h[s], w[s]);
        else
            stencil::su3dag_vec(u, h[s], w[s]);
    }
    // acc += sign (w ; -+ e_mu^dag w), the boundary sign (+-1) folded into
    // fused multiply-adds
#pragma unroll
    for (int c = 0; c < 3; c++) {
        cx<R> a, b;  // e_mu^dag w
        switch (mu) {
            case 0: a = -w[0][c]; b = -w[1][c]; break;
            case 1: a = timesI(w[1][c]); b = timesI(w[0][c]); break;
            case 2: a = w[1][c]; b = -w[0][c]; break;
            default: a = timesI(w[0][c]); b = timesmI(w[1][c]); break;
        }
        if (sgn < 0) {
            a = -a;
            b = -b;
        }
        acc[c].re = fmx(sign, w[0][c].re, acc[c].re);
        acc[c].im = fmx(sign, w[0][c].im, acc[c].im);
        acc[3 + c].re = fmx(sign, w[1][c].re, acc[3 + c].re);
        acc[3 + c].im = fmx(sign, w[1][c].im, acc[3 + c].im);
        acc[6 + c].re = fmx(sign, a.re, acc[6 + c].re);
        acc[6 + c].im = fmx(sign, a.im, acc[6 + c].im);
        acc[9 + c].re = fmx(sign, b.re, acc[9 + c].re);
        acc[9 + c].im = fmx(sign, b.im, acc[9 + c].im);
    }
}

struct SiteInfo {
    long grank;     // global rank
    int x[4];       // global coordinates
    int l[4];       // block-local coordinates
};

__device__ __forceinline__ void block_site(const Geom &g, const BlkGeom &B, const int org[4], int par, int t,
                                           SiteInfo &s)
{
    int row = t / B.bs3h;
    int x3h = t - row * B.bs3h;
    int tt = row / B.bs[2];
    s.l[2] = row - tt * B.bs[2];
    s.l[0] = tt / B.bs[1];
    s.l[1] = tt - s.l[0] * B.bs[1];
    int b = (par + s.l[0] + s.l[1] + s.l[2]) & 1;   // block origin has even parity
    s.l[3] = 2 * x3h + b;
    for (int i = 0; i < 4; i++) s.x[i] = org[i] + s.l[i];
    s.grank = coords_rank(g, s.x);
}

// local rank of the in-block neighbour l + d mu, or -1 if it leaves the block
__device__ __forceinline__ int blk_nbr(const BlkGeom &B, const int l[4], int mu, int d)
{
    int m[4] = {l[0], l[1], l[2], l[3]};
    int v = m[mu] + d;
    if (v < 0 || v >= B.bs[mu]) {
        if (!B.wrap[mu]) return -1;
        v = v < 0 ? v + B.bs[mu] : v - B.bs[mu];
    }
    m[mu] = v;
    return (m[3] + B.bs[3] * (m[2] + B.bs[2] * (m[1] + B.bs[1] * m[0]))) >> 1;
}

// acc = sum of the 8 in-block projected hops of src (parity 1-par) at site s (parity par)
template <class R, class LK>
__device__ void block_hopsum(const Geom &g, const BlkGeom &B, const LK *U, int par, const SiteInfo &s,
                             const cx<R> *src, cx<R> acc[12])
{
#pragma unroll
    for (int i = 0; i < 12; i++) acc[i] = mk(R(0), R(0));
    cx<R> u[3][3], v[12];
    for (int mu = 0; mu < 4; mu++) {
        int lf = blk_nbr(B, s.l, mu, +1);
        if (lf >= 0) {
            R sg = (mu == 0 && s.x[0] == g.L[0] - 1) ? R(g.bc_t) : R(1);
            glink(U, g.Vh, par, mu, s.grank, u);
            sload(src, B.nh, lf, v);
            proj_apply<R>(mu, -1, v, u, false, sg, acc);
        }
        int lb = blk_nbr(B, s.l, mu, -1);
        if (lb >= 0) {
            R sg = (mu == 0 && s.x[0] == 0) ? R(g.bc_t) : R(1);
            int y[4] = {s.x[0], s.x[1], s.x[2], s.x[3]};
            y[mu] = y[mu] == 0 ? g.L[mu] - 1 : y[mu] - 1;
            glink(U, g.Vh, 1 - par, mu, coords_rank(g, y), u);
            sload(src, B.nh, lb, v);
            proj_apply<R>(mu, +1, v, u, true, sg, acc);
        }
    }
}

template <class R>
__device__ __forceinline__ void block_reduce2(R &a, R &b, R &c, R *red)
{
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
        c += __shfl_down_sync(0xffffffffu, c, o);
    }
    int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
    __syncthreads();
    if (lane == 0) {
        red[3 * warp] = a;
        red[3 * warp + 1] = b;
        red[3 * warp + 2] = c;
    }
    __syncthreads();
    a = b = c = 0;
    for (int w = 0; w < nw; w++) {
        a += red[3 * w];
        b += red[3 * w + 1];
        c += red[3 * w + 2];
    }
}

template <int P>
struct SapArgs {
    Geom g;
    BlkGeom B;
    const int *blocks;   // block ids of this colour
    typename SapT<P>::SP *r;        // native full fields (residual; the block's part is replaced)
    typename SapT<P>::SP *psi;      // native full fields (updated)
    typename SapT<P>::SP *delta;    // native full fields: chi of the blocks of this colour
    long fstride;                    // spinor units between the fields of consecutive right-hand sides
    const typename SapT<P>::LK *U;
    const typename SapT<P>::CL *Ae, *Aio;   // A on even sites, A^-1 on odd sites
    // the operator as the resident block kernel reads it: in block order (perm = 1,
    // site t of the block in place slot of the plan's list at slot * nh + t) or,
    // where the copy could not be allocated, the arrays above (perm = 0)
    const typename SapT<P>::LK *Ub;
    const typename SapT<P>::CL *Aeb, *Aiob;
    int perm, slot0;     // slot of block list entry 0
    int nmr;
};

__device__ __forceinline__ void gstore(double2 *f, long Vh, long r, const cx<double> v[12])
{
#pragma unroll
    for (int c = 0; c < 12; c++) f[c * Vh + r] = make_double2(v[c].re, v[c].im);
}
__device__ __forceinline__ void gstore(float4 *f, long Vh, long r, const cx<float> v[12])
{
#pragma unroll
    for (int q = 0; q < 6; q++)
        f[q * Vh + r] = make_float4(v[2 * q].re, v[2 * q].im, v[2 * q + 1].re, v[2 * q + 1].im);
}
__device__ __forceinline__ void gstore(h16s *f, long Vh, long r, const cx<float> v[12]) { f16s_store(f, Vh, r, v); }

constexpr int SAPS_NH = 128;   // sites of one parity per block (4^4 blocks)

template <int P>
__global__ void __launch_bounds__(128) k_sap_block(SapArgs<P> a)
{
    using R = typename SapT<P>::R;
    using SP = typename SapT<P>::SP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const BlkGeom &B = a.B;
    const int nh = B.nh;
    cx<R> *rho = (cx<R> *)smem_raw;
    cx<R> *chi = rho + 12 * nh;
    cx<R> *pv = chi + 12 * nh;
    cx<R> *to = pv + 12 * nh;
    cx<R> *ro = to + 12 * nh;
    R *red = (R *)(ro + 12 * nh);
    const long Vh = a.g.Vh;
    const long half = SapT<P>::half(Vh);
    const long foff = blockIdx.y * a.fstride;
    SP *r_e = a.r + foff, *r_o = a.r + foff + half;
    SP *psi_e = a.psi + foff, *psi_o = a.psi + foff + half;
    SP *d_e = a.delta + foff, *d_o = a.delta + foff + half;

    int bid = a.blocks[blockIdx.x];
    int org[4];
    {
        int t = bid;
        int c3 = t % B.nb[3];
        t /= B.nb[3];
        int c2 = t % B.nb[2];
        t /= B.nb[2];
        int c1 = t % B.nb[1];
        int c0 = t / B.nb[1];
        org[0] = c0 * B.bs[0];
        org[1] = c1 * B.bs[1];
        org[2] = c2 * B.bs[2];
        org[3] = c3 * B.bs[3];
    }
    cx<R> v[12], w[12];
    // r_o into smem, to = A_oo^-1 r_o
    for (int t = threadIdx.x; t < nh; t += blockDim.x) {
        SiteInfo s;
        block_site(a.g, B, org, 1, t, s);
        gload(r_o, Vh, s.grank, v);
        sstore(ro, nh, t, v);
        clov_apply<R>(a.Aio, Vh, s.grank, v, w);
        sstore(to, nh, t, w);
    }
    __syncthreads();
    // rho = b_e = r_e - H_eo,blk to  (H = -1/2 S)
    for (int t = threadIdx.x; t < nh; t += blockDim.x) {
        SiteInfo s;
        block_site(a.g, B, org, 0, t, s);
        gload(r_e, Vh, s.grank, v);
        block_hopsum<R>(a.g, B, a.U, 0, s, to, w);
#pragma unroll
        for (int c = 0; c < 12; c++) {
            v[c] = v[c] + R(0.5) * w[c];
            chi[c * nh + t] = mk(R(0), R(0));
        }
        sstore(rho, nh, t, v);
    }
    __syncthreads();
    for (int it = 0; it < a.nmr; it++) {
        // to = A_oo^-1 H_oe,blk rho
        for (int t = threadIdx.x; t < nh; t += blockDim.x) {
            SiteInfo s;
            block_site(a.g, B, org, 1, t, s);
            block_hopsum<R>(a.g, B, a.U, 1, s, rho, w);
#pragma unroll
            for (int c = 0; c < 12; c++) w[c] = R(-0.5) * w[c];
            clov_apply<R>(a.Aio, Vh, s.grank, w, v);
            sstore(to, nh, t, v);
        }
        __syncthreads();
        // p = A_ee rho - H_eo,blk to
        R pp = 0, pr_re = 0, pr_im = 0;
        for (int t = threadIdx.x; t < nh; t += blockDim.x) {
            SiteInfo s;
            block_site(a.g, B, org, 0, t, s);
            cx<R> x[12];
            sload(rho, nh, t, x);
            clov_apply<R>(a.Ae, Vh, s.grank, x, v);
            block_hopsum<R>(a.g, B, a.U, 0, s, to, w);
#pragma unroll
            for (int c = 0; c < 12; c++) {
                v[c] = v[c] + R(0.5) * w[c];
                pp += v[c].re * v[c].re + v[c].im * v[c].im;
                pr_re += v[c].re * x[c].re + v[c].im * x[c].im;   // conj(p) rho
                pr_im += v[c].re * x[c].im - v[c].im * x[c].re;
            }
            sstore(pv, nh, t, v);
        }
        block_reduce2<R>(pp, pr_re, pr_im, red);
        if (pp == R(0)) break;   // rho = 0: the block is solved
        R ar = pr_re / pp, ai = pr_im / pp;
        cx<R> alpha = mk(ar, ai);
        for (int t = threadIdx.x; t < nh; t += blockDim.x) {
#pragma unroll
            for (int c = 0; c < 12; c++) {
                cx<R> rv = rho[c * nh + t];
                chi[c * nh + t] = chi[c * nh + t] + alpha * rv;
                rho[c * nh + t] = rv - alpha * pv[c * nh + t];
            }
        }
        __syncthreads();
    }
    // chi_o = A_oo^-1 (r_o - H_oe,blk chi_e); psi += chi; delta = chi.
    // The block's new residual r - D_blk chi is (rho, 0): on odd sites it vanishes
    // by construction of chi_o, on even sites it is the MinRes residual of
    // Dhat_blk chi_e = b_e.  Hops from chi into other blocks are applied by
    // k_sap_face_l afterwards.
    for (int t = threadIdx.x; t < nh; t += blockDim.x) {
        SiteInfo s;
        block_site(a.g, B, org, 1, t, s);
        block_hopsum<R>(a.g, B, a.U, 1, s, chi, w);
        sload(ro, nh, t, v);
#pragma unroll
        for (int c = 0; c < 12; c++) v[c] = v[c] + R(0.5) * w[c];
        clov_apply<R>(a.Aio, Vh, s.grank, v, w);
        gadd(psi_o, Vh, s.grank, w);
        gstore(d_o, Vh, s.grank, w);
#pragma unroll
        for (int c = 0; c < 12; c++) w[c] = mk(R(0), R(0));
        gstore(r_o, Vh, s.grank, w);
        SiteInfo se;
        block_site(a.g, B, org, 0, t, se);
        sload(chi, nh, t, v);
        gadd(psi_e, Vh, se.grank, v);
        gstore(d_e, Vh, se.grank, v);
        sload(rho, nh, t, v);
        gstore(r_e, Vh, se.grank, v);
    }
}

// ------------------------------------------------------------------------
// FP64 block solve, four threads a site.
//
// The FP64 pipe bounds it (2 multiply-adds a clock and SM; operands from shared
// memory and L2 have ten times the time they need), so the split is the one with
// the fewest FP64 instructions issued:
//  - thread group mu takes both hops of direction mu, its sites ordered with x_mu
//    slowest: for 4^4 blocks a warp is a plane of constant x_mu, so the hops that
//    leave the block, a quarter of all, are skipped by whole warps;
//  - the backward product is accumulated on top of the forward one, which gives
//    the upper spins w+ + w- without an addition and the lower ones as
//    (w+ + w-) - 2 w+;
//  - signs and factors i are integer operations on the sign bit;
//  - each thread then adds the four directions' shares of one spin (group k owns
//    spin k, through shared memory), applies three rows of the clover block and
//    does the MinRes updates of its three components; the factor -1/2 of the
//    hops between the two parities is applied once, at the end (-1/4).
// All phases are one loop, so that the four directions' code is there once.
// 32 x 16^3, 256 blocks of 4^4 a launch, 5 steps: 862 us (one thread a site: 1268 us), the FP64
// pipe 85 % busy on an SM that has a block; 256 blocks on 152 SMs leave a third of
// the SMs idle in the second half.
struct SapD {
    double2 *X, *rho, *to;   // shares [4][12][nh]; block vectors [12][nh]
    double *red;             // [3][16], then alpha (2) and <p,p>
};
constexpr size_t sap_d_smem(int nh) { return (size_t)72 * nh * sizeof(double2) + 51 * sizeof(double); }

__device__ __forceinline__ double flip_if(bool neg, double v)
{
    return __hiloint2double(__double2hiint(v) ^ (neg ? 0x80000000 : 0), __double2loint(v));
}
__device__ __forceinline__ double minus(double v) { return flip_if(true, v); }

// w += U h (DAG: U^dag h), or w = ... (INIT), for both spins; u points at the
// link's nine entries, Vh apart
template <bool DAG, bool INIT>
__device__ __forceinline__ void d_su3(const double2 *__restrict__ u, long Vh, const cx<double> h[2][3],
                                      cx<double> w[2][3])
{
    double2 m[9];
#pragma unroll
    for (int e = 0; e < 9; e++) m[e] = __ldg(u + e * Vh);
#pragma unroll
    for (int j = 0; j < 3; j++)
#pragma unroll
        for (int i = 0; i < 3; i++) {
            const double2 q = DAG ? m[3 * j + i] : m[3 * i + j];
#pragma unroll
            for (int s = 0; s < 2; s++) {
                const cx<double> x = h[s][j];
                cx<double> &y = w[s][i];
                y.re = INIT && j == 0 ? q.x * x.re : fmx(q.x, x.re, y.re);
                y.re = fmx(DAG ? q.y : -q.y, x.im, y.re);
                y.im = INIT && j == 0 ? q.x * x.im : fmx(q.x, x.im, y.im);
                y.im = fmx(DAG ? -q.y : q.y, x.re, y.im);
            }
        }
}

// projected neighbour spinor, times the time-boundary sign
template <int MU, int SGN>
__device__ __forceinline__ void d_project(const double2 *src, int nh, bool neg, cx<double> h[2][3])
{
    stencil::Spinor<double> v;
#pragma unroll
    for (int c = 0; c < 12; c++) {
        const double2 t = src[c * nh];
        v.s[c / 3][c % 3] = mk(t.x, t.y);
    }
    stencil::project<double, MU, SGN>(v, h);
    if (MU == 0)
#pragma unroll
        for (int i = 0; i < 6; i++)
            h[i / 3][i % 3] = mk(flip_if(neg, h[i / 3][i % 3].re), flip_if(neg, h[i / 3][i % 3].im));
}

// Share of direction MU in the hop sum (before the -1/2) of one site, into
// X[MU][.][t].  nf, nb: slots of the neighbours in src, or -1; uf, ub: the links.
template <int MU>
__device__ __forceinline__ void d_hops(const double2 *uf, const double2 *ub, long Vh, const double2 *src, int nh,
                                       int nf, int nb, bool negf, bool negb, double2 *X)
{
    cx<double> h[2][3], w[2][3], d[2][3];
    if (nf >= 0) {
        d_project<MU, -1>(src + nf, nh, negf, h);
        d_su3<false, true>(uf, Vh, h, w);
        if (nb >= 0) {
            cx<double> f[2][3];
#pragma unroll
            for (int i = 0; i < 6; i++) f[i / 3][i % 3] = w[i / 3][i % 3];
            d_project<MU, 1>(src + nb, nh, negb, h);
            d_su3<true, false>(ub, Vh, h, w);
#pragma unroll
            for (int i = 0; i < 6; i++) {
                const cx<double> a = f[i / 3][i % 3], b = w[i / 3][i % 3];
                d[i / 3][i % 3] = mk(fmx(-2.0, a.re, b.re), fmx(-2.0, a.im, b.im));
            }
        } else {
#pragma unroll
            for (int i = 0; i < 6; i++) {
                const cx<double> a = w[i / 3][i % 3];
                d[i / 3][i % 3] = mk(minus(a.re), minus(a.im));
            }
        }
    } else if (nb >= 0) {
        d_project<MU, 1>(src + nb, nh, negb, h);
        d_su3<true, true>(ub, Vh, h, w);
#pragma unroll
        for (int i = 0; i < 6; i++) d[i / 3][i % 3] = w[i / 3][i % 3];
    } else {
#pragma unroll
        for (int i = 0; i < 6; i++) w[i / 3][i % 3] = d[i / 3][i % 3] = mk(0.0, 0.0);
    }
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const cx<double> a = d[0][c], b = d[1][c];
        double2 l0, l1;   // e_mu^dag d
        switch (MU) {
            case 0:
                l0 = make_double2(minus(a.re), minus(a.im));
                l1 = make_double2(minus(b.re), minus(b.im));
                break;
            case 1:
                l0 = make_double2(minus(b.im), b.re);
                l1 = make_double2(minus(a.im), a.re);
                break;
            case 2:
                l0 = make_double2(b.re, b.im);
                l1 = make_double2(minus(a.re), minus(a.im));
                break;
            default:
                l0 = make_double2(minus(a.im), a.re);
                l1 = make_double2(b.im, minus(b.re));
                break;
        }
        X[c * nh] = make_double2(w[0][c].re, w[0][c].im);
        X[(3 + c) * nh] = make_double2(w[1][c].re, w[1][c].im);
        X[(6 + c) * nh] = l0;
        X[(9 + c) * nh] = l1;
    }
}

// rows 3 HALF .. 3 HALF + 2 of a packed Hermitian 6x6 block (entries Vh apart)
// times in[0..5] (nh apart)
template <int HALF>
__device__ __forceinline__ void d_rows(const double2 *__restrict__ A, long Vh, const double2 *in, int nh,
                                       cx<double> out[3])
{
    const double2 d0 = __ldg(A + (HALF ? 1 : 0) * Vh), d1 = __ldg(A + (HALF ? 2 : 1) * Vh);
    const double dg[3] = {HALF ? d0.y : d0.x, HALF ? d1.x : d0.y, HALF ? d1.y : d1.x};
    cx<double> v[6];
#pragma unroll
    for (int i = 0; i < 6; i++) v[i] = mk(in[i * nh].x, in[i * nh].y);
#pragma unroll
    for (int i = 0; i < 3; i++) out[i] = mk(dg[i] * v[3 * HALF + i].re, dg[i] * v[3 * HALF + i].im);
    int k = 3;
#pragma unroll
    for (int i = 0; i < 6; i++)
#pragma unroll
        for (int j = i + 1; j < 6; j++, k++) {
            const bool ri = i / 3 == HALF, rj = j / 3 == HALF;
            if (!ri && !rj) continue;
            const double2 o = __ldg(A + k * Vh);
            if (ri) {   // out_i += o v_j
                cx<double> &y = out[i - 3 * HALF];
                y.re = fmx(o.x, v[j].re, y.re);
                y.re = fmx(-o.y, v[j].im, y.re);
                y.im = fmx(o.x, v[j].im, y.im);
                y.im = fmx(o.y, v[j].re, y.im);
            }
            if (rj) {   // out_j += conj(o) v_i
                cx<double> &y = out[j - 3 * HALF];
                y.re = fmx(o.x, v[i].re, y.re);
                y.re = fmx(o.y, v[i].im, y.re);
                y.im = fmx(o.x, v[i].im, y.im);
                y.im = fmx(-o.y, v[i].re, y.im);
            }
        }
}

// Site i (0 .. nh-1) of parity par with x_mu slowest, and its neighbours along mu
struct SapDSite {
    int t, rank, nf, nb, rb;   // slot, global rank, neighbours' slots or -1, rank of the backward one
    bool negf, negb;           // time-boundary sign of the two hops
};
__device__ __forceinline__ SapDSite d_site(const Geom &g, const BlkGeom &B, const int org[4], int mu, int par, int i)
{
    const int last = mu == 3 ? 2 : 3, hl = B.bs[last] >> 1;   // the direction halved by parity
    int l[4], r = i / hl, sum = par;
    const int lh = i - r * hl;
#pragma unroll
    for (int m = 3; m >= 0; m--) {
        if (m == last || m == mu) continue;
        l[m] = r % B.bs[m];
        r /= B.bs[m];
        sum += l[m];
    }
    l[mu] = r;
    l[last] = 2 * lh + ((sum + r) & 1);
    int x[4];
#pragma unroll
    for (int m = 0; m < 4; m++) x[m] = org[m] + l[m];
    SapDSite s;
    s.t = (l[3] + B.bs[3] * (l[2] + B.bs[2] * (l[1] + B.bs[1] * l[0]))) >> 1;
    s.rank = (int)coords_rank(g, x);
    s.nf = blk_nbr(B, l, mu, 1);
    s.nb = blk_nbr(B, l, mu, -1);
    s.negf = mu == 0 && x[0] == g.L[0] - 1 && g.bc_t < 0;
    s.negb = mu == 0 && x[0] == 0 && g.bc_t < 0;
    x[mu] = x[mu] == 0 ? g.L[mu] - 1 : x[mu] - 1;
    s.rb = (int)coords_rank(g, x);
    return s;
}

__global__ void __launch_bounds__(4 * SAPS_NH, 1) k_sap_block_d(SapArgs<LQCD_F64> a)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const BlkGeom &B = a.B;
    const int nh = B.nh, gs = blockDim.x >> 2;
    SapD S;
    S.X = (double2 *)smem_raw;
    S.rho = S.X + 48 * nh;
    S.to = S.rho + 12 * nh;
    S.red = (double *)(S.to + 12 * nh);
    const long Vh = a.g.Vh;
    const long half = 12 * Vh, foff = blockIdx.y * a.fstride;
    const int k = threadIdx.x / gs, i = threadIdx.x - k * gs;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool act = i < nh;
    int org[4];
    {
        int q = a.blocks[blockIdx.x];
#pragma unroll
        for (int m = 3; m >= 0; m--) {
            org[m] = q % B.nb[m] * B.bs[m];
            q /= B.nb[m];
        }
    }
    const SapDSite so = d_site(a.g, B, org, k, 1, act ? i : 0), se = d_site(a.g, B, org, k, 0, act ? i : 0);
    // three components of spin k of the two parities
    const long co = 3 * k * Vh + so.rank, ce = 3 * k * Vh + se.rank;
    cx<double> chi[3], s[3], w[3];
#pragma unroll
    for (int j = 0; j < 3; j++) chi[j] = s[j] = w[j] = mk(0.0, 0.0);
    const int last = 2 * a.nmr + 1;
    //   ph = -1            to = A_oo^-1 r_o
    //   ph = 0             rho = r_e - H_eo to = r_e + 1/2 S(to)
    //   odd ph < last      to = A_oo^-1 S(rho) = -2 A_oo^-1 H_oe rho
    //   even ph            p = A_ee rho - 1/4 S(to); the MinRes step
    //   ph = last          chi_o = A_oo^-1 (r_o + 1/2 S(chi_e)), chi_e read from to
#pragma unroll 1
    for (int ph = -1; ph <= last; ph++) {
        const bool odd = ph & 1;
        const int t = odd ? so.t : se.t;
        if (ph >= 0) {
            if (act) {
                const double2 *src = odd && ph < last ? S.rho : S.to;
                const int nf = odd ? so.nf : se.nf, nb = odd ? so.nb : se.nb;
                const bool negf = odd ? so.negf : se.negf, negb = odd ? so.negb : se.negb;
                const double2 *uf = a.U + (long)((odd * 4 + k) * 9) * Vh + (odd ? so.rank : se.rank);
                const double2 *ub = a.U + (long)((!odd * 4 + k) * 9) * Vh + (odd ? so.rb : se.rb);
                double2 *X = S.X + 12 * k * nh + t;
                switch (k) {
                    case 0: d_hops<0>(uf, ub, Vh, src, nh, nf, nb, negf, negb, X); break;
                    case 1: d_hops<1>(uf, ub, Vh, src, nh, nf, nb, negf, negb, X); break;
                    case 2: d_hops<2>(uf, ub, Vh, src, nh, nf, nb, negf, negb, X); break;
                    default: d_hops<3>(uf, ub, Vh, src, nh, nf, nb, negf, negb, X); break;
                }
            }
            __syncthreads();
            if (act)
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    const double2 *x = S.X + (3 * k + j) * nh + t;
                    const double2 x0 = x[0], x1 = x[12 * nh], x2 = x[24 * nh], x3 = x[36 * nh];
                    s[j] = mk(((x0.x + x1.x) + x2.x) + x3.x, ((x0.y + x1.y) + x2.y) + x3.y);
                }
        }
        bool fin = ph == last - 1;   // the next phase is the last
        if (ph == 0) {
            if (act)
#pragma unroll
                for (int j = 0; j < 3; j++) {
                    const double2 r = a.r[foff + ce + j * Vh];
                    S.rho[(3 * k + j) * nh + t] = make_double2(fmx(0.5, s[j].re, r.x), fmx(0.5, s[j].im, r.y));
                }
        } else {
            // input of the clover rows: rho itself, or the odd phases' sum by way of
            // X, whose entries of this site and spin no other thread reads
            if (odd) {
                if (act)
#pragma unroll
                    for (int j = 0; j < 3; j++) {
                        if (ph < 0 || ph == last) {
                            const double2 r = a.r[foff + half + co + j * Vh];
                            s[j] = mk(fmx(0.5, s[j].re, r.x), fmx(0.5, s[j].im, r.y));
                        }
                        S.X[(3 * k + j) * nh + t] = make_double2(s[j].re, s[j].im);
                    }
                __syncthreads();
            }
            if (act) {
                const double2 *in = (odd ? S.X : S.rho) + 6 * (k >> 1) * nh + t;
                const double2 *A = (odd ? a.Aio : a.Ae) + (long)(18 * (k >> 1)) * Vh + (odd ? so.rank : se.rank);
                if (k & 1)
                    d_rows<1>(A, Vh, in, nh, w);
                else
                    d_rows<0>(A, Vh, in, nh, w);
            }
            if (odd) {
                if (act && ph < last)
#pragma unroll
                    for (int j = 0; j < 3; j++) S.to[(3 * k + j) * nh + t] = make_double2(w[j].re, w[j].im);
            } else {
                double dot[4] = {0, 0, 0, 0};   // <p,p>, <p,rho>
                cx<double> rv[3];
                if (act)
#pragma unroll
                    for (int j = 0; j < 3; j++) {
                        const double2 r = S.rho[(3 * k + j) * nh + t];
                        rv[j] = mk(r.x, r.y);
                        w[j] = mk(fmx(-0.25, s[j].re, w[j].re), fmx(-0.25, s[j].im, w[j].im));
                        dot[0] = fmx(w[j].im, w[j].im, fmx(w[j].re, w[j].re, dot[0]));
                        dot[1] = fmx(w[j].im, r.y, fmx(w[j].re, r.x, dot[1]));
                        dot[2] = fmx(-w[j].im, r.x, fmx(w[j].re, r.y, dot[2]));
                    }
                warp_multi_sum<4>(dot);
                if ((lane & 7) == 0 && lane < 24) S.red[16 * (lane >> 3) + warp] = dot[0];
                __syncthreads();
                if (warp == 0) {
                    const bool has = lane < (int)(blockDim.x >> 5);
                    double f[4] = {has ? S.red[lane] : 0, has ? S.red[16 + lane] : 0, has ? S.red[32 + lane] : 0, 0};
                    warp_multi_sum<4>(f);
                    const double pp = __shfl_sync(0xffffffffu, f[0], 0);
                    if (lane == 0) S.red[50] = pp;
                    if ((lane == 8 || lane == 16) && pp != 0) S.red[47 + lane / 8] = f[0] / pp;
                }
                __syncthreads();
                if (S.red[50] == 0) {   // rho = 0: the block is solved
                    fin = true;
                    ph = last - 1;
                } else if (act) {
                    const double ar = S.red[48], ai = S.red[49];
#pragma unroll
                    for (int j = 0; j < 3; j++) {
                        // chi += alpha rho, rho -= alpha p
                        chi[j].re = fmx(-ai, rv[j].im, fmx(ar, rv[j].re, chi[j].re));
                        chi[j].im = fmx(ai, rv[j].re, fmx(ar, rv[j].im, chi[j].im));
                        S.rho[(3 * k + j) * nh + t] = make_double2(fmx(ai, w[j].im, fmx(-ar, w[j].re, rv[j].re)),
                                                                   fmx(-ai, w[j].re, fmx(-ar, w[j].im, rv[j].im)));
                    }
                }
            }
        }
        if (fin && act)
#pragma unroll
            for (int j = 0; j < 3; j++) S.to[(3 * k + j) * nh + se.t] = make_double2(chi[j].re, chi[j].im);
        __syncthreads();
    }
    // psi += chi; delta = chi; r <- (rho, 0), as in k_sap_block
    if (act)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const long e = foff + ce + j * Vh, o = foff + half + co + j * Vh;
            const double2 pe = a.psi[e], po = a.psi[o];
            a.psi[e] = make_double2(pe.x + chi[j].re, pe.y + chi[j].im);
            a.psi[o] = make_double2(po.x + w[j].re, po.y + w[j].im);
            a.delta[e] = make_double2(chi[j].re, chi[j].im);
            a.delta[o] = make_double2(w[j].re, w[j].im);
            a.r[e] = S.rho[(3 * k + j) * nh + se.t];
            a.r[o] = make_double2(0.0, 0.0);
        }
}

// ------------------------------------------------------------------------
// FP32 block solve with the whole block resident in shared memory.
//
// At the start of a block visit the CTA stages the block's forward links (two
// rows, all sites and directions), A_ee on its even sites, A_oo^-1 on its odd
// sites and r_o into shared memory with coalesced loads; all MinRes phases
// then run from shared memory.  Two threads per site: in a hop phase thread
// h = 0 sums the four forward hops and h = 1 the four backward hops, the pair
// exchanges its partial sums by a lane shuffle, and each thread then applies
// one chirality block (spins 2h, 2h+1) of the clover term.  Same arithmetic
// as k_sap_block, different summation order.

// Shared memory of the resident block kernel.  SA: the clover term of the
// block is staged too (172 KB, one CTA per SM); without it every clover
// application reads its 6x6 block through L1/L2 (same values) and two FP32
// CTAs (98 KB) or three F16S CTAs (74 KB: the links kept in FP16, the
// precision they are stored in) fit on an SM.  The MinRes correction chi stays
// in registers (each thread owns its half-site) and goes through p at the end.
// staging loads: one 4-real word of a link row pair or of the clover term
__device__ __forceinline__ float4 stage4(const float4 *p) { return __ldg(p); }
__device__ __forceinline__ float4 stage4(const uint2 *p)
{
    uint2 t = __ldg(p);
    cx<float> a = f16s_h2c(t.x, 1.f), b = f16s_h2c(t.y, 1.f);
    return make_float4(a.re, a.im, b.re, b.im);
}
__device__ __forceinline__ void stage_link(float4 &d, const float4 *p) { d = __ldg(p); }
__device__ __forceinline__ void stage_link(float4 &d, const uint2 *p) { d = stage4(p); }
__device__ __forceinline__ void stage_link(uint2 &d, const uint2 *p) { d = __ldg(p); }
__device__ __forceinline__ float4 link4(float4 v) { return v; }
__device__ __forceinline__ float4 link4(uint2 t)
{
    cx<float> a = f16s_h2c(t.x, 1.f), b = f16s_h2c(t.y, 1.f);
    return make_float4(a.re, a.im, b.re, b.im);
}
struct SapSmemA {
    float4 U[4][3][2 * SAPS_NH];   // forward links, two rows, site par * SAPS_NH + t
    float4 A[18][2 * SAPS_NH];     // A (even sites) or A^-1 (odd sites), site par * SAPS_NH + t
    float4 rho[6][SAPS_NH], p[6][SAPS_NH], to[6][SAPS_NH], ro[6][SAPS_NH];
    float red[3][8];
};
struct SapSmemL {
    float4 U[4][3][2 * SAPS_NH];
    float4 rho[6][SAPS_NH], p[6][SAPS_NH], to[6][SAPS_NH], ro[6][SAPS_NH];
    float red[3][8];
};
struct SapSmemH {
    uint2 U[4][3][2 * SAPS_NH];    // FP16 link rows
    float4 rho[6][SAPS_NH], p[6][SAPS_NH], to[6][SAPS_NH], ro[6][SAPS_NH];
    float red[3][8];
};
template <int P, bool SA>
using SapSmem = std::conditional_t<SA, SapSmemA, std::conditional_t<P == LQCD_F16S, SapSmemH, SapSmemL>>;
// resident CTAs per SM of each layout (the launch bounds)
template <int P, bool SA>
constexpr int sap_ctas() { return SA ? 1 : (P == LQCD_F16S ? 3 : 2); }

__device__ __forceinline__ int blk_lex(const BlkGeom &B, const int l[4])
{
    return l[3] + B.bs[3] * (l[2] + B.bs[2] * (l[1] + B.bs[1] * l[0]));
}

// local lexicographic index of the in-block neighbour l + d mu, or -1
__device__ __forceinline__ int blk_nbr_lex(const BlkGeom &B, const int l[4], int mu, int d)
{
    int m[4] = {l[0], l[1], l[2], l[3]};
    int v = m[mu] + d;
    if (v < 0 || v >= B.bs[mu]) {
        if (!B.wrap[mu]) return -1;
        v = v < 0 ? v + B.bs[mu] : v - B.bs[mu];
    }
    m[mu] = v;
    return blk_lex(B, m);
}

__device__ __forceinline__ void s_spinor(const float4 (*f)[SAPS_NH], int t, cx<float> v[12])
{
#pragma unroll
    for (int q = 0; q < 6; q++) {
        float4 a = f[q][t];
        v[2 * q] = mk(a.x, a.y);
        v[2 * q + 1] = mk(a.z, a.w);
    }
}
template <class SM>
__device__ __forceinline__ void s_link(const SM &S, int mu, int ls, cx<float> u[3][3])
{
#pragma unroll
    for (int q = 0; q < 3; q++) {
        const float4 a = link4(S.U[mu][q][ls]);
        u[(2 * q) / 3][(2 * q) % 3] = mk(a.x, a.y);
        u[(2 * q + 1) / 3][(2 * q + 1) % 3] = mk(a.z, a.w);
    }
    su3_third_row(u);
}
// one chirality block h of the clover matrix applied to v[6]; the block is
// read from shared memory (local site ls) or from global memory (rank grank)
template <bool SA, class SM, class CL>
__device__ __forceinline__ void s_clover_half(const SM &S, int ls, const CL *A, long Vh, long grank, int h,
                                              const cx<float> v[6], cx<float> w[6])
{
    float a[36];
#pragma unroll
    for (int q = 0; q < 9; q++) {
        float4 t;
        if constexpr (SA)
            t = S.A[9 * h + q][ls];
        else
            t = stage4(A + (9 * h + q) * Vh + grank);
        a[4 * q] = t.x;
        a[4 * q + 1] = t.y;
        a[4 * q + 2] = t.z;
        a[4 * q + 3] = t.w;
    }
    stencil::Herm6<float> hm;
#pragma unroll
    for (int i = 0; i < 6; i++) hm.d[i] = a[i];
#pragma unroll
    for (int i = 0; i < 15; i++) hm.o[i] = mk(a[6 + 2 * i], a[7 + 2 * i]);
    stencil::herm_apply(hm, v, w);
}

// projected hop of direction mu in either sense with the sense a runtime value:
// sgn = -1 (forward, 1 - gamma_mu) or +1 (backward, 1 + gamma_mu), u already
// the matrix to apply (U or U^dag).  The arithmetic of proj_apply with the
// same sense: the signs enter as exact factors of fused multiply-adds, so the
// two threads of a site pair (one per sense) run one instruction stream.
template <int MU>
__device__ __forceinline__ void proj_apply_rt(float sgn, const cx<float> psi[12], const cx<float> u[3][3], float sign,
                                              cx<float> acc[12])
{
    cx<float> h[2][3], w[2][3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const cx<float> u0 = psi[c], u1 = psi[3 + c], l0 = psi[6 + c], l1 = psi[9 + c];
        cx<float> el0, el1;
        switch (MU) {
            case 0: el0 = -l0; el1 = -l1; break;
            case 1: el0 = timesmI(l1); el1 = timesmI(l0); break;
            case 2: el0 = -l1; el1 = l0; break;
            default: el0 = timesmI(l0); el1 = timesI(l1); break;
        }
        h[0][c] = mk(fmx(sgn, el0.re, u0.re), fmx(sgn, el0.im, u0.im));
        h[1][c] = mk(fmx(sgn, el1.re, u1.re), fmx(sgn, el1.im, u1.im));
    }
    stencil::su3_vec(u, h[0], w[0]);
    stencil::su3_vec(u, h[1], w[1]);
    const float ss = sign * sgn;
#pragma unroll
    for (int c = 0; c < 3; c++) {
        cx<float> a, b;
        switch (MU) {
            case 0: a = -w[0][c]; b = -w[1][c]; break;
            case 1: a = timesI(w[1][c]); b = timesI(w[0][c]); break;
            case 2: a = w[1][c]; b = -w[0][c]; break;
            default: a = timesI(w[0][c]); b = timesmI(w[1][c]); break;
        }
        acc[c].re = fmx(sign, w[0][c].re, acc[c].re);
        acc[c].im = fmx(sign, w[0][c].im, acc[c].im);
        acc[3 + c].re = fmx(sign, w[1][c].re, acc[3 + c].re);
        acc[3 + c].im = fmx(sign, w[1][c].im, acc[3 + c].im);
        acc[6 + c].re = fmx(ss, a.re, acc[6 + c].re);
        acc[6 + c].im = fmx(ss, a.im, acc[6 + c].im);
        acc[9 + c].re = fmx(ss, b.re, acc[9 + c].re);
        acc[9 + c].im = fmx(ss, b.im, acc[9 + c].im);
    }
}

// Chirality half h of the in-block hop sum S (before the -1/2) at site (l, x)
// from the smem field src of the other parity: thread h = 0 takes the forward
// hops, h = 1 the backward ones, each hands the other's half over and adds what
// it gets to its own.  own: the site's index par * SAPS_NH + t in the link
// arrays; the neighbours' links sit at (1 - par) * SAPS_NH + their half index.
// Both threads run the same instructions (the sense, the link slot and U versus
// U^dag are selected per lane), and a hop that leaves the block is computed
// with weight 0 instead of being skipped, so the warp never diverges here; its
// dummy neighbour is t itself, the neighbour of a lane nearby, so that the
// loads stay free of bank conflicts.
template <class SM>
__device__ __forceinline__ void s_hopsum(const Geom &g, const BlkGeom &B, const SM &S, int h, const int l[4],
                                         const int x[4], int own, const float4 (*src)[SAPS_NH], cx<float> out[6])
{
    cx<float> acc[12];
#pragma unroll
    for (int i = 0; i < 12; i++) acc[i] = mk(0.f, 0.f);
    const float sgn = h ? 1.f : -1.f;
    const int d = h ? -1 : 1;
    const int oth = own < SAPS_NH ? SAPS_NH : 0, t = own < SAPS_NH ? own : own - SAPS_NH;
    const int xt = h ? 0 : g.L[0] - 1;
    cx<float> u[3][3], v[12];
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        const int ln = blk_nbr_lex(B, l, mu, d);
        const int n = ln >= 0 ? ln >> 1 : t;
        float sg = (mu == 0 && x[0] == xt) ? float(g.bc_t) : 1.f;
        sg = ln >= 0 ? sg : 0.f;
        s_link(S, mu, h ? oth + n : own, u);
        cx<float> m[3][3];
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int k = 0; k < 3; k++) m[a][k] = h ? mk(u[k][a].re, -u[k][a].im) : u[a][k];
        s_spinor(src, n, v);
        switch (mu) {
            case 0: proj_apply_rt<0>(sgn, v, m, sg, acc); break;
            case 1: proj_apply_rt<1>(sgn, v, m, sg, acc); break;
            case 2: proj_apply_rt<2>(sgn, v, m, sg, acc); break;
            default: proj_apply_rt<3>(sgn, v, m, sg, acc); break;
        }
    }
#pragma unroll
    for (int i = 0; i < 6; i++) {
        const cx<float> give = h ? acc[i] : acc[6 + i], keep = h ? acc[6 + i] : acc[i];
        out[i].re = keep.re + __shfl_xor_sync(0xffffffffu, give.re, 16);
        out[i].im = keep.im + __shfl_xor_sync(0xffffffffu, give.im, 16);
    }
}

__device__ __forceinline__ void stage_site(const float4 *f, long Vh, long r, float4 o[6])
{
#pragma unroll
    for (int q = 0; q < 6; q++) o[q] = f[q * Vh + r];
}
__device__ __forceinline__ void stage_site(const h16s *f, long Vh, long r, float4 o[6])
{
    cx<float> v[12];
    f16s_load<false>(f, Vh, r, v);
#pragma unroll
    for (int q = 0; q < 6; q++) o[q] = make_float4(v[2 * q].re, v[2 * q].im, v[2 * q + 1].re, v[2 * q + 1].im);
}
// chirality half h (components 6h .. 6h+5) of site r.  The F16S forms are
// called by both threads of a site pair (lanes l and l ^ 16) together: the
// pair agrees on the site's scale through a lane shuffle.
__device__ __forceinline__ void half_load(const float4 *f, long Vh, long r, int h, cx<float> v[6])
{
#pragma unroll
    for (int q = 0; q < 3; q++) {
        float4 a = f[(3 * h + q) * Vh + r];
        v[2 * q] = mk(a.x, a.y);
        v[2 * q + 1] = mk(a.z, a.w);
    }
}
__device__ __forceinline__ void half_store(float4 *f, long Vh, long r, int h, const cx<float> v[6])
{
#pragma unroll
    for (int q = 0; q < 3; q++) f[(3 * h + q) * Vh + r] = make_float4(v[2 * q].re, v[2 * q].im, v[2 * q + 1].re, v[2 * q + 1].im);
}
__device__ __forceinline__ void half_load(const h16s *f, long Vh, long r, int h, cx<float> v[6])
{
    // h = 0: components 0..3 (uint4 0) and 4, 5 (low half of uint4 1);
    // h = 1: components 6, 7 (high half of uint4 1) and 8..11 (uint4 2)
    const uint4 *q = reinterpret_cast<const uint4 *>(f);
    const float sc = f16s_scales(f, Vh)[r];
    const uint2 mid = reinterpret_cast<const uint2 *>(q + Vh + r)[h];
    const uint4 end = q[(h ? 2 : 0) * Vh + r];
    const cx<float> a0 = f16s_h2c(end.x, sc), a1 = f16s_h2c(end.y, sc), a2 = f16s_h2c(end.z, sc),
                    a3 = f16s_h2c(end.w, sc), m0 = f16s_h2c(mid.x, sc), m1 = f16s_h2c(mid.y, sc);
    v[0] = h ? m0 : a0;
    v[1] = h ? m1 : a1;
    v[2] = h ? a0 : a2;
    v[3] = h ? a1 : a3;
    v[4] = h ? a2 : m0;
    v[5] = h ? a3 : m1;
}
__device__ __forceinline__ void half_store(h16s *f, long Vh, long r, int h, const cx<float> v[6])
{
    float m = 0.f;
#pragma unroll
    for (int i = 0; i < 6; i++) m = fmaxf(m, fmaxf(fabsf(v[i].re), fabsf(v[i].im)));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    const float inv = f16s_inv(m);
    uint4 *q = reinterpret_cast<uint4 *>(f);
    const cx<float> e0 = h ? v[2] : v[0], e1 = h ? v[3] : v[1], e2 = h ? v[4] : v[2], e3 = h ? v[5] : v[3];
    const cx<float> m0 = h ? v[0] : v[4], m1 = h ? v[1] : v[5];
    q[(h ? 2 : 0) * Vh + r] = make_uint4(f16s_c2h(e0, inv), f16s_c2h(e1, inv), f16s_c2h(e2, inv), f16s_c2h(e3, inv));
    reinterpret_cast<uint2 *>(q + Vh + r)[h] = make_uint2(f16s_c2h(m0, inv), f16s_c2h(m1, inv));
    if (h == 0) f16s_scales(f, Vh)[r] = m;
}
template <class SP>
__device__ __forceinline__ void half_add(SP *f, long Vh, long r, int h, const cx<float> v[6])
{
    cx<float> t[6];
    half_load(f, Vh, r, h, t);
#pragma unroll
    for (int i = 0; i < 6; i++) t[i] = t[i] + v[i];
    half_store(f, Vh, r, h, t);
}

// block list entry bi of a.blocks, right-hand side rhs; blockDim.x = 2 nh.  DEP: the
// kernel may have been launched dependently.
template <int P, bool SA, bool DEP>
__device__ __forceinline__ void sap_block_s_body(const SapArgs<P> &a, int bi, int rhs)
{
    using SP = typename SapT<P>::SP;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SapSmem<P, SA> &S = *reinterpret_cast<SapSmem<P, SA> *>(smem_raw);
    const BlkGeom &B = a.B;
    const int nh = B.nh;
    const long Vh = a.g.Vh;
    const long half = SapT<P>::half(Vh);
    const long foff = rhs * a.fstride;
    SP *r_e = a.r + foff, *r_o = a.r + foff + half;
    SP *psi_e = a.psi + foff, *psi_o = a.psi + foff + half;
    SP *d_e = a.delta + foff, *d_o = a.delta + foff + half;
    int org[4];
    {
        int t = a.blocks[bi];
        int c3 = t % B.nb[3];
        t /= B.nb[3];
        int c2 = t % B.nb[2];
        t /= B.nb[2];
        int c1 = t % B.nb[1];
        int c0 = t / B.nb[1];
        org[0] = c0 * B.bs[0];
        org[1] = c1 * B.bs[1];
        org[2] = c2 * B.bs[2];
        org[3] = c3 * B.bs[3];
    }
    const int tid = threadIdx.x;
    const typename SapT<P>::LK *U = a.perm ? a.Ub : a.U;
    const typename SapT<P>::CL *Ae = a.perm ? a.Aeb : a.Ae, *Aio = a.perm ? a.Aiob : a.Aio;
    const long op0 = (long)(a.slot0 + bi) * nh;   // the block's first site in the block-ordered operator
    // ---- stage links and clover, then r_o and r_e (one thread per block site, both
    // parities); the operator is constant, r is the work of the kernel before
    for (int i = tid; i < 2 * nh; i += blockDim.x) {
        const int par = i >= nh, t = par ? i - nh : i;
        SiteInfo s;
        if (!a.perm) block_site(a.g, B, org, par, t, s);
        const int ls = par * SAPS_NH + t;
        const long op = a.perm ? op0 + t : s.grank;
#pragma unroll
        for (int mu = 0; mu < 4; mu++)
#pragma unroll
            for (int q = 0; q < 3; q++) stage_link(S.U[mu][q][ls], U + ((long)(par * 4 + mu) * 3 + q) * Vh + op);
        if constexpr (SA) {
            const typename SapT<P>::CL *A = par ? Aio : Ae;
#pragma unroll
            for (int q = 0; q < 18; q++) S.A[q][ls] = stage4(A + q * Vh + op);
        }
    }
    if constexpr (DEP) after_previous();
    for (int i = tid; i < 2 * nh; i += blockDim.x) {
        const int par = i >= nh, t = par ? i - nh : i;
        SiteInfo s;
        block_site(a.g, B, org, par, t, s);
        float4 site[6];
        stage_site(par ? r_o : r_e, Vh, s.grank, site);
        if (par) {
#pragma unroll
            for (int q = 0; q < 6; q++) S.ro[q][t] = site[q];
        } else {
#pragma unroll
            for (int q = 0; q < 6; q++) S.rho[q][t] = site[q];
        }
    }
    __syncthreads();
    // chirality half / hop direction h and site rank t: lanes 0-15 of a warp
    // take h = 0 of 16 sites, lanes 16-31 h = 1 of the same sites, so the 8
    // lanes of every quarter-warp read consecutive rows of one shared-memory
    // array (no bank conflicts between a site's two halves)
    const int h = (tid >> 4) & 1, t = ((tid >> 5) << 4) | (tid & 15);
    const bool act = t < nh;
    SiteInfo so = {}, se = {};
    const int lso = SAPS_NH + t, lse = t;   // the sites' slots in the link / clover arrays
    if (act) {
        block_site(a.g, B, org, 1, t, so);
        block_site(a.g, B, org, 0, t, se);
    }
    const long opo = a.perm ? op0 + t : so.grank, ope = a.perm ? op0 + t : se.grank;
    cx<float> ah[6], v[6], w[6];
    float4 chi4[3];   // this thread's half of chi_e
#pragma unroll
    for (int q = 0; q < 3; q++) chi4[q] = make_float4(0.f, 0.f, 0.f, 0.f);
    // to = A_oo^-1 r_o (chirality half h)
    if (act) {
#pragma unroll
        for (int q = 0; q < 3; q++) {
            float4 x = S.ro[3 * h + q][t];
            v[2 * q] = mk(x.x, x.y);
            v[2 * q + 1] = mk(x.z, x.w);
        }
        s_clover_half<SA>(S, lso, Aio, Vh, opo, h, v, w);
#pragma unroll
        for (int q = 0; q < 3; q++) S.to[3 * h + q][t] = make_float4(w[2 * q].re, w[2 * q].im, w[2 * q + 1].re, w[2 * q + 1].im);
    }
    __syncthreads();
    // rho = r_e - H_eo to = r_e + 1/2 S
    if (act) {
        s_hopsum(a.g, B, S, h, se.l, se.x, lse, S.to, ah);
#pragma unroll
        for (int q = 0; q < 3; q++) {
            float4 x = S.rho[3 * h + q][t];
            const cx<float> s0 = ah[2 * q], s1 = ah[2 * q + 1];
            S.rho[3 * h + q][t] = make_float4(x.x + 0.5f * s0.re, x.y + 0.5f * s0.im, x.z + 0.5f * s1.re, x.w + 0.5f * s1.im);
        }
    }
    __syncthreads();
    for (int it = 0; it < a.nmr; it++) {
        // to = A_oo^-1 (-1/2 S(rho))
        if (act) {
            s_hopsum(a.g, B, S, h, so.l, so.x, lso, S.rho, ah);
#pragma unroll
            for (int i = 0; i < 6; i++) v[i] = -0.5f * ah[i];
            s_clover_half<SA>(S, lso, Aio, Vh, opo, h, v, w);
#pragma unroll
            for (int q = 0; q < 3; q++) S.to[3 * h + q][t] = make_float4(w[2 * q].re, w[2 * q].im, w[2 * q + 1].re, w[2 * q + 1].im);
        }
        __syncthreads();
        // p = A_ee rho + 1/2 S(to); partial <p,p>, <p,rho>
        float pp = 0.f, pr = 0.f, pi = 0.f;
        if (act) {
            s_hopsum(a.g, B, S, h, se.l, se.x, lse, S.to, ah);
            cx<float> x[6];
#pragma unroll
            for (int q = 0; q < 3; q++) {
                float4 y = S.rho[3 * h + q][t];
                x[2 * q] = mk(y.x, y.y);
                x[2 * q + 1] = mk(y.z, y.w);
            }
            s_clover_half<SA>(S, lse, Ae, Vh, ope, h, x, w);
#pragma unroll
            for (int i = 0; i < 6; i++) {
                w[i] = w[i] + 0.5f * ah[i];
                pp += w[i].re * w[i].re + w[i].im * w[i].im;
                pr += w[i].re * x[i].re + w[i].im * x[i].im;
                pi += w[i].re * x[i].im - w[i].im * x[i].re;
            }
#pragma unroll
            for (int q = 0; q < 3; q++) S.p[3 * h + q][t] = make_float4(w[2 * q].re, w[2 * q].im, w[2 * q + 1].re, w[2 * q + 1].im);
        }
        for (int o = 16; o > 0; o >>= 1) {
            pp += __shfl_down_sync(0xffffffffu, pp, o);
            pr += __shfl_down_sync(0xffffffffu, pr, o);
            pi += __shfl_down_sync(0xffffffffu, pi, o);
        }
        if ((tid & 31) == 0) {
            S.red[0][tid >> 5] = pp;
            S.red[1][tid >> 5] = pr;
            S.red[2][tid >> 5] = pi;
        }
        __syncthreads();
        pp = pr = pi = 0.f;
        for (int wv = 0; wv < (int)(blockDim.x >> 5); wv++) {
            pp += S.red[0][wv];
            pr += S.red[1][wv];
            pi += S.red[2][wv];
        }
        __syncthreads();
        if (pp == 0.f) break;   // rho = 0: the block is solved
        const float ar = pr / pp, ai = pi / pp;
        if (act) {
#pragma unroll
            for (int q = 0; q < 3; q++) {
                float4 rv = S.rho[3 * h + q][t], pv = S.p[3 * h + q][t], cv = chi4[q];
                // chi += alpha rho, rho -= alpha p
                cv.x += ar * rv.x - ai * rv.y;
                cv.y += ar * rv.y + ai * rv.x;
                cv.z += ar * rv.z - ai * rv.w;
                cv.w += ar * rv.w + ai * rv.z;
                rv.x -= ar * pv.x - ai * pv.y;
                rv.y -= ar * pv.y + ai * pv.x;
                rv.z -= ar * pv.z - ai * pv.w;
                rv.w -= ar * pv.w + ai * pv.z;
                chi4[q] = cv;
                S.rho[3 * h + q][t] = rv;
            }
        }
        __syncthreads();
    }
    // chi_o = A_oo^-1 (r_o + 1/2 S(chi_e)); psi += chi; delta = chi; r <- (rho, 0)
    // (chi_e goes to the block through p, which is free now)
    if (act)
#pragma unroll
        for (int q = 0; q < 3; q++) S.p[3 * h + q][t] = chi4[q];
    __syncthreads();
    if (act) {
        s_hopsum(a.g, B, S, h, so.l, so.x, lso, S.p, ah);
#pragma unroll
        for (int q = 0; q < 3; q++) {
            float4 x = S.ro[3 * h + q][t];
            v[2 * q] = mk(x.x + 0.5f * ah[2 * q].re, x.y + 0.5f * ah[2 * q].im);
            v[2 * q + 1] = mk(x.z + 0.5f * ah[2 * q + 1].re, x.w + 0.5f * ah[2 * q + 1].im);
        }
        s_clover_half<SA>(S, lso, Aio, Vh, opo, h, v, w);
        cx<float> ce[6], re[6], zero[6];
#pragma unroll
        for (int q = 0; q < 3; q++) {
            const float4 c4 = chi4[q], r4 = S.rho[3 * h + q][t];
            ce[2 * q] = mk(c4.x, c4.y);
            ce[2 * q + 1] = mk(c4.z, c4.w);
            re[2 * q] = mk(r4.x, r4.y);
            re[2 * q + 1] = mk(r4.z, r4.w);
            zero[2 * q] = zero[2 * q + 1] = mk(0.f, 0.f);
        }
        half_add(psi_o, Vh, so.grank, h, w);
        half_store(d_o, Vh, so.grank, h, w);
        half_store(r_o, Vh, so.grank, h, zero);
        half_add(psi_e, Vh, se.grank, h, ce);
        half_store(d_e, Vh, se.grank, h, ce);
        half_store(r_e, Vh, se.grank, h, re);
    }
}

template <int P, bool SA>
__global__ void __launch_bounds__(2 * SAPS_NH, sap_ctas<P, SA>()) k_sap_block_s(SapArgs<P> a)
{
    sap_block_s_body<P, SA, true>(a, blockIdx.x, blockIdx.y);
}

// LQCD_SAP_STAGE_A = 0 | 1 forces the clover term through L1 or staged in
// shared memory (test instrumentation); otherwise the autotuner chooses.
// Returns -1 when not forced.
int sap_stage_forced()
{
    const char *e = getenv("LQCD_SAP_STAGE_A");
    if (!e || !*e) return -1;
    return e[0] == '1' ? 1 : 0;
}

// r(x) -= sum of the hops into x from neighbours y that lie in another block of
// colour col (delta holds chi there), over a precomputed list of the sites that
// receive such hops: entry (i, mask) with i the parity-major site index and bit
// 2 mu + (d > 0) of mask set for each hop from x + d mu.  The list is sorted by
// mask, so the threads of a warp take the same hops (a thread per lattice site
// branches per site and took twice the time).
template <int P>
__device__ __forceinline__ void sap_face_site(const SapArgs<P> &a, int2 fs, int rhs)
{
    using R = typename SapT<P>::R;
    using SP = typename SapT<P>::SP;
    const long Vh = a.g.Vh;
    const int par = fs.x >= Vh;
    const long rk = par ? fs.x - Vh : fs.x;
    const long half = SapT<P>::half(Vh);
    const long foff = rhs * a.fstride;
    int x[4];
    rank_coords(a.g, par, (int)rk, x);
    cx<R> acc[12], u[3][3], v[12];
#pragma unroll
    for (int c = 0; c < 12; c++) acc[c] = mk(R(0), R(0));
    const SP *din = a.delta + foff + (1 - par) * half;
    for (int mu = 0; mu < 4; mu++)
        for (int d = -1; d <= 1; d += 2) {
            if (!((fs.y >> (2 * mu + (d > 0))) & 1)) continue;
            const long ry = nbr_rank(a.g, x, mu, d);
            gload(din, Vh, ry, v);
            if (d > 0) {
                R sg = (mu == 0 && x[0] == a.g.L[0] - 1) ? R(a.g.bc_t) : R(1);
                glink(a.U, Vh, par, mu, rk, u);
                proj_apply<R>(mu, -1, v, u, false, sg, acc);
            } else {
                R sg = (mu == 0 && x[0] == 0) ? R(a.g.bc_t) : R(1);
                glink(a.U, Vh, 1 - par, mu, ry, u);
                proj_apply<R>(mu, +1, v, u, true, sg, acc);
            }
        }
    // r -= H delta = r + 1/2 S
#pragma unroll
    for (int c = 0; c < 12; c++) acc[c] = R(0.5) * acc[c];
    gadd(a.r + foff + par * half, Vh, rk, acc);
}
template <int P>
__global__ void __launch_bounds__(128) k_sap_face_l(SapArgs<P> a, const int2 *__restrict__ list, int n)
{
    const long e = blockIdx.x * (long)blockDim.x + threadIdx.x;
    const int2 fs = list[min(e, n - 1L)];
    after_previous();
    if (e < n) sap_face_site<P>(a, fs, blockIdx.y);
}

// ------------------------------------------------------------------ batches
// Several lattices in one launch.  args[2 l + col]: the SAP arguments of
// lattice l for the blocks of colour col.  Persistent CTAs take work items from
// a device counter (*queue, zero before the launch) until the list is empty;
// items of lattices whose active flag is 0 are skipped.
template <int P, bool SA>
__global__ void __launch_bounds__(2 * SAPS_NH, sap_ctas<P, SA>())
    k_sap_block_s_batch(const SapArgs<P> *args, int col, const int2 *items, int nitems, const int *active, int *queue)
{
    __shared__ int s_item;
    __shared__ SapArgs<P> sa;
    for (;;) {
        if (threadIdx.x == 0) s_item = atomicAdd(queue, 1);
        __syncthreads();
        const int it = s_item;
        if (it >= nitems) return;
        const int2 w = items[it];   // (lattice, index in its list of colour col)
        const bool on = !active || active[w.x];
        if (on && threadIdx.x == 0) sa = args[2 * w.x + col];
        __syncthreads();
        if (on) sap_block_s_body<P, SA, false>(sa, w.y, 0);
        __syncthreads();
    }
}

// items: (lattice, first list entry of a tile of up to 128, entries in the tile);
// lists[2 l + col]: the face list of lattice l after colour col
template <int P>
__global__ void __launch_bounds__(128)
    k_sap_face_batch(const SapArgs<P> *args, int col, const int2 *const *lists, const int4 *items, const int *active)
{
    const int4 w = items[blockIdx.x];
    if (active && !active[w.x]) return;
    __shared__ SapArgs<P> sa;
    if (threadIdx.x == 0) sa = args[2 * w.x + col];
    __syncthreads();
    if ((int)threadIdx.x < w.z) sap_face_site<P>(sa, lists[2 * w.x + col][w.y + threadIdx.x], 0);
}

// LQCD_SAP_GENERIC=1 selects the generic (L1-cached) FP32 block kernel
bool sap_force_generic()
{
    const char *e = getenv("LQCD_SAP_GENERIC");
    return e && e[0] == '1';
}

struct SapPlan {
    int bs[4] = {0, 0, 0, 0};
    int *blocks_dev = nullptr;   // [colour 0 ids..., colour 1 ids...]
    int count[2] = {0, 0};
    BlkGeom B;
    int2 *face_dev[2] = {nullptr, nullptr};   // sites updated after colour col (k_sap_face_l)
    int nface[2] = {0, 0};
    // the operator in block order, [F32, F16S]: links, A_ee, A_oo^-1 in one buffer
    // (the plan's own; made again when the context's operator has changed)
    struct Perm {
        void *p = nullptr;
        long version = -1;
        bool failed = false;
    } perm[2];
};

// one cached plan per context (keyed by block shape)
struct PlanCache {
    lqcd_ctx *ctx;
    SapPlan plan;
};
std::list<PlanCache> g_plans;   // a list: pointers to its plans stay valid as it grows

lqcd_status get_plan(lqcd_ctx *c, const int bs[4], SapPlan **out)
{
    for (auto &pc : g_plans)
        if (pc.ctx == c && pc.plan.bs[0] == bs[0] && pc.plan.bs[1] == bs[1] && pc.plan.bs[2] == bs[2] &&
            pc.plan.bs[3] == bs[3]) {
            *out = &pc.plan;
            return LQCD_OK;
        }
    SapPlan P;
    int vol = 1;
    for (int i = 0; i < 4; i++) {
        if (bs[i] <= 0 || bs[i] % 2 || c->g.L[i] % bs[i])
            return set_err(c, LQCD_ERR_ARG, "block extent %d does not tile L[%d]=%d", bs[i], i, c->g.L[i]);
        P.bs[i] = bs[i];
        P.B.bs[i] = bs[i];
        P.B.nb[i] = c->g.L[i] / bs[i];
        P.B.wrap[i] = P.B.nb[i] == 1;
        vol *= bs[i];
    }
    if (vol / 2 > 1024) return set_err(c, LQCD_ERR_ARG, "SAP block of %d sites too large", vol);
    P.B.nh = vol / 2;
    P.B.bs3h = bs[3] / 2;
    std::vector<int> ids[2];
    for (int c0 = 0; c0 < P.B.nb[0]; c0++)
        for (int c1 = 0; c1 < P.B.nb[1]; c1++)
            for (int c2 = 0; c2 < P.B.nb[2]; c2++)
                for (int c3 = 0; c3 < P.B.nb[3]; c3++) {
                    int id = c3 + P.B.nb[3] * (c2 + P.B.nb[2] * (c1 + P.B.nb[1] * c0));
                    ids[(c0 + c1 + c2 + c3) & 1].push_back(id);
                }
    P.count[0] = (int)ids[0].size();
    P.count[1] = (int)ids[1].size();
    std::vector<int> all(ids[0]);
    all.insert(all.end(), ids[1].begin(), ids[1].end());
    LQCD_CUDA_CHECK(c, cudaMalloc(&P.blocks_dev, all.size() * sizeof(int)));
    LQCD_CUDA_CHECK(c, cudaMemcpy(P.blocks_dev, all.data(), all.size() * sizeof(int), cudaMemcpyHostToDevice));
    // face lists: for each site, the hops that enter from a block of colour col
    // (a different block; both parities, parity-major index), sorted by hop mask
    {
        const int *L = c->g.L;
        const long Vh = c->g.Vh;
        std::vector<std::pair<int, int>> fl[2];   // (mask, index)
        int x[4];
        for (x[0] = 0; x[0] < L[0]; x[0]++)
            for (x[1] = 0; x[1] < L[1]; x[1]++)
                for (x[2] = 0; x[2] < L[2]; x[2]++)
                    for (x[3] = 0; x[3] < L[3]; x[3]++) {
                        const long lex = x[3] + (long)L[3] * (x[2] + (long)L[2] * (x[1] + (long)L[1] * x[0]));
                        const int par = (x[0] + x[1] + x[2] + x[3]) & 1;
                        const int idx = (int)(par * Vh + (lex >> 1));
                        int bx[4], bsum = 0;
                        for (int m = 0; m < 4; m++) {
                            bx[m] = x[m] / bs[m];
                            bsum += bx[m];
                        }
                        int mask[2] = {0, 0};
                        for (int mu = 0; mu < 4; mu++)
                            for (int d = -1; d <= 1; d += 2) {
                                int y = x[mu] + d;
                                y = y < 0 ? y + L[mu] : (y >= L[mu] ? y - L[mu] : y);
                                const int by = y / bs[mu];
                                if (by == bx[mu]) continue;
                                mask[(bsum - bx[mu] + by) & 1] |= 1 << (2 * mu + (d > 0));
                            }
                        for (int col = 0; col < 2; col++)
                            if (mask[col]) fl[col].push_back({mask[col], idx});
                    }
        for (int col = 0; col < 2; col++) {
            std::sort(fl[col].begin(), fl[col].end());
            std::vector<int2> h(fl[col].size());
            for (size_t k = 0; k < h.size(); k++) h[k] = make_int2(fl[col][k].second, fl[col][k].first);
            P.nface[col] = (int)h.size();
            if (h.empty()) continue;
            LQCD_CUDA_CHECK(c, cudaMalloc(&P.face_dev[col], h.size() * sizeof(int2)));
            LQCD_CUDA_CHECK(c, cudaMemcpy(P.face_dev[col], h.data(), h.size() * sizeof(int2), cudaMemcpyHostToDevice));
        }
    }
    g_plans.push_back({c, P});
    *out = &g_plans.back().plan;
    return LQCD_OK;
}

// row-wise copy out[row Vh + slot nh + t] = in[row Vh + rank], rows of parity par0 +
// row / rows_per_parity
template <class T>
__global__ void k_sap_permute(Geom g, BlkGeom B, const int *blocks, int rows_per_parity, int par0,
                              const T *__restrict__ in, T *out)
{
    const long pos = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (pos >= g.Vh) return;
    const int row = blockIdx.y, par = par0 + row / rows_per_parity;
    const int slot = (int)(pos / B.nh), t = (int)(pos - (long)slot * B.nh);
    int id = blocks[slot], org[4];
#pragma unroll
    for (int i = 3; i >= 0; i--) {
        org[i] = id % B.nb[i] * B.bs[i];
        id /= B.nb[i];
    }
    SiteInfo s;
    block_site(g, B, org, par, t, s);
    out[row * (long)g.Vh + pos] = in[row * (long)g.Vh + s.grank];
}

// The block-ordered operator of the plan, in args.  A block's 128 sites per
// parity lie in runs of bs3 / 2 ranks, so that a warp's load of one link or
// clover word touched 16 lines: at nmr = 4 the clover loads alone were 40 % of
// the L1 wavefronts that bounded the kernel (67 % of their peak).  In block
// order they are one run.  With the halved lane exchange of s_hopsum, per colour
// launch at 32 x 16^3: F16S, 12 right-hand sides, nmr 4: 444 -> 380 us; FP32, one,
// nmr 5: 64.5 -> 49.4 us.
template <int P>
lqcd_status sap_operator(lqcd_ctx *c, SapPlan &pl, SapArgs<P> &a)
{
    using LK = typename SapT<P>::LK;
    using CL = typename SapT<P>::CL;
    static_assert(sizeof(LK) == sizeof(CL), "one buffer");
    const long Vh = c->g.Vh;
    SapPlan::Perm &pm = pl.perm[P == LQCD_F32 ? 0 : 1];
    a.perm = 0;
    a.Ub = a.U;
    a.Aeb = a.Ae;
    a.Aiob = a.Aio;
    // A caller's graph reads the lattice-ordered arrays (the same bits): replayed after
    // the links have changed it would find the copy of the operator it was captured
    // with, and a copy recorded here would not be made before the next eager call.
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(c->stream, &cap) != cudaSuccess) {
        cudaGetLastError();   // the legacy stream, while another one is captured
        cap = cudaStreamCaptureStatusNone;
    }
    if (cap != cudaStreamCaptureStatusNone) return LQCD_OK;
    if (!pm.p && !pm.failed) {
        if (cudaMalloc(&pm.p, (24 + 2 * 18) * Vh * sizeof(LK)) != cudaSuccess) {
            cudaGetLastError();
            pm.p = nullptr;
            pm.failed = true;   // the lattice-ordered arrays serve
        }
    }
    if (!pm.p) return LQCD_OK;
    LK *ub = (LK *)pm.p;
    CL *ae = (CL *)(ub + 24 * Vh), *ai = ae + 18 * Vh;
    if (pm.version != c->op_version) {
        const int gx = div_up(Vh, 256);
        k_sap_permute<LK><<<dim3(gx, 24), 256, 0, c->stream>>>(c->g, pl.B, pl.blocks_dev, 12, 0, a.U, ub);
        k_sap_permute<CL><<<dim3(gx, 18), 256, 0, c->stream>>>(c->g, pl.B, pl.blocks_dev, 18, 0, a.Ae, ae);
        k_sap_permute<CL><<<dim3(gx, 18), 256, 0, c->stream>>>(c->g, pl.B, pl.blocks_dev, 18, 1, a.Aio, ai);
        c->n_kernel_launches += 3;
        LQCD_LAUNCH_CHECK(c);
        pm.version = c->op_version;
    }
    a.perm = 1;
    a.Ub = ub;
    a.Aeb = ae;
    a.Aiob = ai;
    return LQCD_OK;
}

template <int P>
lqcd_status sap_run(lqcd_ctx *c, SapPlan &P_, int ncy, int nmr, const void *eta, void *psi, void *r,
                    void *delta, int nrhs)
{
    using T = SapT<P>;
    using R = typename T::R;
    using SP = typename T::SP;
    SapPlan &Pl = P_;
    const size_t fb = 2 * native_half_bytes(c, (lqcd_prec)P);
    size_t smem = 5 * 12 * Pl.B.nh * sizeof(cx<R>) + 3 * 32 * sizeof(R);
    static bool attr_set = false;
    if (!attr_set) {
        cudaFuncSetAttribute(k_sap_block<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
        attr_set = true;
    }
    if (smem > 200 * 1024) return set_err(c, LQCD_ERR_ARG, "SAP block needs %zu bytes of shared memory", smem);
    if (nrhs < 1 || nrhs > 65535) return set_err(c, LQCD_ERR_ARG, "SAP nrhs=%d", nrhs);
    LQCD_CUDA_CHECK(c, cudaMemsetAsync(psi, 0, fb * nrhs, c->stream));
    LQCD_CUDA_CHECK(c, cudaMemcpyAsync(r, eta, fb * nrhs, cudaMemcpyDeviceToDevice, c->stream));
    SapArgs<P> a;
    a.g = c->g;
    a.B = Pl.B;
    a.r = (SP *)r;
    a.psi = (SP *)psi;
    a.delta = (SP *)delta;
    a.fstride = 2 * T::half(c->g.Vh);
    if constexpr (P == LQCD_F64) {
        a.U = c->U64;
        a.Ae = c->A64[0];
        a.Aio = c->Ai64[1];
    } else if constexpr (P == LQCD_F32) {
        a.U = c->U32;
        a.Ae = c->A32[0];
        a.Aio = c->Ai32[1];
    } else {
        a.U = c->U16;
        a.Ae = c->A16[0];
        a.Aio = c->Ai16[1];
    }
    a.nmr = nmr;
    int threads = std::min(128, Pl.B.nh);
    // FP32 / F16S with blocks of <= 128 sites per parity (whole warps of site
    // pairs): the shared-memory resident kernel
    bool resident = false;
    // FP64 with blocks of <= 128 sites per parity: four threads a site (512 of 128
    // registers at most); larger ones one thread a site in turns
    const bool four = P == LQCD_F64 && Pl.B.nh <= SAPS_NH && !sap_force_generic();
    if constexpr (P == LQCD_F64) {
        static bool attr_d = false;
        if (!attr_d) {
            cudaFuncSetAttribute(k_sap_block_d, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sap_d_smem(SAPS_NH));
            attr_d = true;
        }
    }
    if constexpr (P != LQCD_F64) {
        static bool attr_s = false;
        if (!attr_s) {
            cudaFuncSetAttribute(k_sap_block_s<P, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(SapSmem<P, true>));
            cudaFuncSetAttribute(k_sap_block_s<P, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)sizeof(SapSmem<P, false>));
            attr_s = true;
        }
        resident = Pl.B.nh <= SAPS_NH && (2 * Pl.B.nh) % 32 == 0 && !sap_force_generic();
        if (resident) LQCD_TRY(sap_operator<P>(c, Pl, a));
    }
    // clover term staged in shared memory (stage = 1, one CTA per SM) or read
    // through L1 (stage = 0): identical arithmetic, chosen by timing.  Without
    // a recorded choice the sweeps of this application alternate between the
    // two forms (in-flight tuning: every sweep is part of the result, so the
    // search costs no extra work) and the faster one is recorded.
    int stage = 0;
    bool tuning = false;
    std::string key;
    float best_us[2] = {1e30f, 1e30f};
    cudaEvent_t ev[2] = {nullptr, nullptr};
    if (P != LQCD_F64 && resident) {
        const int forced = sap_stage_forced();
        if (forced >= 0) {
            stage = forced;
        } else {
            key = tune_key(c, (std::string("k_sap_block_s/b") + std::to_string(Pl.bs[0]) + "x" +
                               std::to_string(Pl.bs[1]) + "x" + std::to_string(Pl.bs[2]) + "x" +
                               std::to_string(Pl.bs[3])).c_str(),
                           0, P, nrhs);
            TuneChoice tc;
            if (tune_lookup(key, &tc)) {
                stage = tc.variant;
            } else if (tune_enabled() && ncy * (Pl.count[1] > 0 ? 2 : 1) >= 4) {
                tuning = true;
                LQCD_CUDA_CHECK(c, cudaEventCreate(&ev[0]));
                LQCD_CUDA_CHECK(c, cudaEventCreate(&ev[1]));
            }
        }
    }
    // the residual is not needed after the last sweep
    int last_col = Pl.count[1] > 0 ? 1 : 0;
    int sweep = 0;
    // Dependent launches hide launch and staging, a part of a short sweep's time, but the
    // CTAs set up early go to the SMs that the kernel before leaves first.  Eight steps of
    // a GCR, 4 x 5 sweeps each, dependent / plain, by CTAs a sweep: FP32 8 to 128 0.90 to
    // 0.93, 192 to 400 0.96 to 1.03 (0.98 at 32 x 16^3, one field), 576 to 6000 0.99 to 1.03;
    // F16S (three CTAs an SM, so the packing is the tightest) 8 to 128 0.91 to 0.93, 192 0.97
    // to 1.00, 243 1.22, 256 1.20, 384 to 6000 1.02 to 1.10.  FP64 (faces only): 0.996.
    const long sweep_ctas = (long)std::max(Pl.count[0], Pl.count[1]) * nrhs;
    const bool dependent = !c->capturing && sweep_ctas <= (P == LQCD_F16S ? 152 : 3 * 152);
    for (int cyc = 0; cyc < ncy; cyc++)
        for (int col = 0; col < 2; col++) {
            if (Pl.count[col] == 0) continue;
            a.slot0 = col == 0 ? 0 : Pl.count[0];
            a.blocks = Pl.blocks_dev + a.slot0;
            if (tuning) {
                stage = (sweep + 1) & 1;   // sweep 0 (cold caches) uses stage 1, then alternate
                cudaEventRecord(ev[0], c->stream);
            }
            if constexpr (P != LQCD_F64) {
                // (the first may follow the kernels that make the operator's copy, whose
                // writes it would stage too early)
                const bool pdl = dependent && sweep > 0;
                if (resident && stage)
                    launch_pdl_smem(pdl, k_sap_block_s<P, true>, dim3(Pl.count[col], nrhs), 2 * Pl.B.nh,
                                    sizeof(SapSmem<P, true>), c->stream, a);
                else if (resident)
                    launch_pdl_smem(pdl, k_sap_block_s<P, false>, dim3(Pl.count[col], nrhs), 2 * Pl.B.nh,
                                    sizeof(SapSmem<P, false>), c->stream, a);
                else
                    k_sap_block<P><<<dim3(Pl.count[col], nrhs), threads, smem, c->stream>>>(a);
            } else if (four) {
                k_sap_block_d<<<dim3(Pl.count[col], nrhs), 4 * ((Pl.B.nh + 31) & ~31), sap_d_smem(Pl.B.nh), c->stream>>>(a);
            } else {
                k_sap_block<P><<<dim3(Pl.count[col], nrhs), threads, smem, c->stream>>>(a);
            }
            c->n_kernel_launches++;
            LQCD_LAUNCH_CHECK(c);
            if (tuning) {
                cudaEventRecord(ev[1], c->stream);
                LQCD_CUDA_CHECK(c, cudaEventSynchronize(ev[1]));
                float ms = 0;
                cudaEventElapsedTime(&ms, ev[0], ev[1]);
                if (sweep > 0) best_us[stage] = std::min(best_us[stage], 1000.f * ms);
                if (tune_verbose())
                    fprintf(stderr, "tune %s: stage=%d sweep %d %.1f us\n", key.c_str(), stage, sweep, 1000.f * ms);
            }
            sweep++;
            if (cyc == ncy - 1 && col == last_col) continue;
            if (Pl.nface[col] > 0)
                launch_pdl(dependent, k_sap_face_l<P>, dim3(div_up(Pl.nface[col], 128), nrhs), 128, c->stream, a,
                           (const int2 *)Pl.face_dev[col], Pl.nface[col]);
            c->n_kernel_launches++;
            LQCD_LAUNCH_CHECK(c);
        }
    if (tuning) {
        cudaEventDestroy(ev[0]);
        cudaEventDestroy(ev[1]);
        TuneChoice tc;
        tc.variant = best_us[1] < best_us[0] ? 1 : 0;
        tc.tx = 2 * Pl.B.nh;
        tc.ty = 1;
        tc.us = best_us[tc.variant];
        tune_store(key, tc);
    }
    return LQCD_OK;
}

}  // namespace

lqcd_status sap_apply(lqcd_ctx *c, const lqcd_sap_params *sp, const void *eta, void *psi, int nrhs)
{
    if (!c->have_clover) return set_err(c, LQCD_ERR_STATE, "clover term not built");
    if (sp->ncy < 1 || sp->nmr < 0) return set_err(c, LQCD_ERR_ARG, "bad SAP cycle counts");
    SapPlan *P;
    LQCD_TRY(get_plan(c, sp->bs, &P));
    void *r;
    const size_t fb = 2 * native_half_bytes(c, sp->prec);
    LQCD_TRY(ws_get(c, WS_SAP_R, 2 * fb * nrhs, &r));
    void *delta = (char *)r + fb * nrhs;
    if (sp->prec == LQCD_F64) return sap_run<LQCD_F64>(c, *P, sp->ncy, sp->nmr, eta, psi, r, delta, nrhs);
    if (sp->prec == LQCD_F32) return sap_run<LQCD_F32>(c, *P, sp->ncy, sp->nmr, eta, psi, r, delta, nrhs);
    if (sp->prec == LQCD_F16S) return sap_run<LQCD_F16S>(c, *P, sp->ncy, sp->nmr, eta, psi, r, delta, nrhs);
    return set_err(c, LQCD_ERR_ARG, "SAP precision %d not supported", (int)sp->prec);
}

// ------------------------------------------------------------------ batches
struct SapBatch {
    lqcd_prec p = LQCD_F16S;
    int ncy = 4, nmr = 5, nh = 0, nsm = 0;
    void *args = nullptr;                  // SapArgs<p>[2 nlat]
    int2 *blk[2] = {nullptr, nullptr};     // (lattice, index in its colour list)
    int nblk[2] = {0, 0};
    const int2 **lists = nullptr;          // [2 nlat] face lists (the plans' own)
    int4 *face[2] = {nullptr, nullptr};    // (lattice, first list entry, entries) per colour
    int nface[2] = {0, 0};
    int *queue = nullptr;                  // one work counter per block launch of an application
    void *r = nullptr, *psi = nullptr, *delta = nullptr;
};

void sap_batch_free(SapBatch *b)
{
    if (!b) return;
    cudaFree(b->args);
    cudaFree(b->blk[0]);
    cudaFree(b->blk[1]);
    cudaFree(b->lists);
    cudaFree(b->face[0]);
    cudaFree(b->face[1]);
    cudaFree(b->queue);
    delete b;
}

namespace {
template <int P>
lqcd_status sap_batch_args(lqcd_ctx *hc, lqcd_ctx *const *ctx, int n, const lqcd_sap_params *sp, SapBatch *b,
                           const long *off)
{
    using SP = typename SapT<P>::SP;
    std::vector<SapArgs<P>> v;
    std::vector<int2> it[2];
    std::vector<int4> face[2];
    std::vector<const int2 *> lists;
    for (int l = 0; l < n; l++) {
        SapPlan *pl;
        LQCD_TRY(get_plan(ctx[l], sp->bs, &pl));
        if (b->nh == 0) b->nh = pl->B.nh;
        if (pl->B.nh != b->nh || b->nh > SAPS_NH || (2 * b->nh) % 32)
            return set_err(hc, LQCD_ERR_ARG, "batched SAP needs one block shape of <= %d sites per parity", SAPS_NH);
        for (int col = 0; col < 2; col++) {
            SapArgs<P> a;
            a.g = ctx[l]->g;
            a.B = pl->B;
            a.slot0 = col == 0 ? 0 : pl->count[0];
            a.blocks = pl->blocks_dev + a.slot0;
            a.r = (SP *)b->r + off[l];
            a.psi = (SP *)b->psi + off[l];
            a.delta = (SP *)b->delta + off[l];
            a.fstride = 0;
            if constexpr (P == LQCD_F32) {
                a.U = ctx[l]->U32;
                a.Ae = ctx[l]->A32[0];
                a.Aio = ctx[l]->Ai32[1];
            } else {
                a.U = ctx[l]->U16;
                a.Ae = ctx[l]->A16[0];
                a.Aio = ctx[l]->Ai16[1];
            }
            a.nmr = sp->nmr;
            LQCD_TRY(sap_operator<P>(ctx[l], *pl, a));
            LQCD_CUDA_CHECK(hc, cudaStreamSynchronize(ctx[l]->stream));   // the batch runs on its own stream
            v.push_back(a);
            for (int i = 0; i < pl->count[col]; i++) it[col].push_back(make_int2(l, i));
            lists.push_back(pl->face_dev[col]);
            for (int e = 0; e < pl->nface[col]; e += 128)
                face[col].push_back(make_int4(l, e, std::min(128, pl->nface[col] - e), 0));
        }
    }
    LQCD_CUDA_CHECK(hc, cudaMalloc(&b->args, v.size() * sizeof(v[0])));
    LQCD_CUDA_CHECK(hc, cudaMemcpy(b->args, v.data(), v.size() * sizeof(v[0]), cudaMemcpyHostToDevice));
    for (int col = 0; col < 2; col++) {
        b->nblk[col] = (int)it[col].size();
        LQCD_CUDA_CHECK(hc, cudaMalloc(&b->blk[col], std::max<size_t>(1, it[col].size()) * sizeof(int2)));
        LQCD_CUDA_CHECK(hc, cudaMemcpy(b->blk[col], it[col].data(), it[col].size() * sizeof(int2), cudaMemcpyHostToDevice));
    }
    LQCD_CUDA_CHECK(hc, cudaMalloc((void **)&b->lists, lists.size() * sizeof(lists[0])));
    LQCD_CUDA_CHECK(hc, cudaMemcpy((void *)b->lists, lists.data(), lists.size() * sizeof(lists[0]),
                                   cudaMemcpyHostToDevice));
    for (int col = 0; col < 2; col++) {
        b->nface[col] = (int)face[col].size();
        LQCD_CUDA_CHECK(hc, cudaMalloc(&b->face[col], std::max<size_t>(1, face[col].size()) * sizeof(int4)));
        LQCD_CUDA_CHECK(hc, cudaMemcpy(b->face[col], face[col].data(), face[col].size() * sizeof(int4),
                                       cudaMemcpyHostToDevice));
    }
    return LQCD_OK;
}

template <int P>
lqcd_status sap_batch_run(lqcd_ctx *hc, SapBatch *b, const int *active)
{
    static bool attr = false;
    if (!attr) {
        cudaFuncSetAttribute(k_sap_block_s_batch<P, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(SapSmem<P, true>));
        cudaFuncSetAttribute(k_sap_block_s_batch<P, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)sizeof(SapSmem<P, false>));
        attr = true;
    }
    // the batched sweeps are replayed from captured graphs, so no in-flight
    // tuning here: the clover term goes through L1 (two to three CTAs per SM,
    // the work queue's balance) unless the staged form is forced
    const bool sa = sap_stage_forced() == 1;
    const auto *args = (const SapArgs<P> *)b->args;
    const int last_col = b->nblk[1] > 0 ? 1 : 0;
    for (int cyc = 0; cyc < b->ncy; cyc++)
        for (int col = 0; col < 2; col++) {
            if (b->nblk[col] == 0) continue;
            if (sa)
                k_sap_block_s_batch<P, true><<<std::min(b->nblk[col], b->nsm), 2 * b->nh, sizeof(SapSmem<P, true>),
                                               hc->stream>>>(args, col, b->blk[col], b->nblk[col], active,
                                                             b->queue + 2 * cyc + col);
            else
                k_sap_block_s_batch<P, false><<<std::min(b->nblk[col], sap_ctas<P, false>() * b->nsm), 2 * b->nh,
                                                sizeof(SapSmem<P, false>), hc->stream>>>(
                    args, col, b->blk[col], b->nblk[col], active, b->queue + 2 * cyc + col);
            hc->n_kernel_launches++;
            LQCD_LAUNCH_CHECK(hc);
            if (cyc == b->ncy - 1 && col == last_col) continue;
            if (b->nface[col] == 0) continue;
            k_sap_face_batch<P><<<b->nface[col], 128, 0, hc->stream>>>(args, col, b->lists, b->face[col], active);
            hc->n_kernel_launches++;
            LQCD_LAUNCH_CHECK(hc);
        }
    return LQCD_OK;
}
}  // namespace

lqcd_status sap_batch_create(lqcd_ctx *hc, lqcd_ctx *const *ctx, int n, const lqcd_sap_params *sp, void *r,
                             void *psi, void *delta, const long *off, SapBatch **out_b)
{
    if (sp->prec != LQCD_F32 && sp->prec != LQCD_F16S)
        return set_err(hc, LQCD_ERR_ARG, "batched SAP runs in F32 or F16S");
    if (sp->ncy < 1 || sp->nmr < 0) return set_err(hc, LQCD_ERR_ARG, "bad SAP cycle counts");
    SapBatch *b = new SapBatch();
    b->p = sp->prec;
    b->ncy = sp->ncy;
    b->nmr = sp->nmr;
    b->r = r;
    b->psi = psi;
    b->delta = delta;
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&b->nsm, cudaDevAttrMultiProcessorCount, dev);
    lqcd_status st = sp->prec == LQCD_F32 ? sap_batch_args<LQCD_F32>(hc, ctx, n, sp, b, off)
                                          : sap_batch_args<LQCD_F16S>(hc, ctx, n, sp, b, off);
    if (st == LQCD_OK && cudaMalloc(&b->queue, 2 * sp->ncy * sizeof(int)) != cudaSuccess) {
        cudaGetLastError();
        st = set_err(hc, LQCD_ERR_NOMEM, "batched SAP work counters");
    }
    if (st != LQCD_OK) {
        sap_batch_free(b);
        return st;
    }
    *out_b = b;
    return LQCD_OK;
}

// the block-ordered operators of lattices whose operator changed since the batch
// was made, on the contexts' streams (the kernel arguments keep their pointers)
lqcd_status sap_batch_refresh(SapBatch *b, lqcd_ctx *const *ctx, int n, const int bs[4])
{
    for (int l = 0; l < n; l++) {
        SapPlan *pl;
        LQCD_TRY(get_plan(ctx[l], bs, &pl));
        auto again = [&](auto tag) -> lqcd_status {
            constexpr int P = decltype(tag)::value;
            SapArgs<P> a;
            if constexpr (P == LQCD_F32) {
                a.U = ctx[l]->U32;
                a.Ae = ctx[l]->A32[0];
                a.Aio = ctx[l]->Ai32[1];
            } else {
                a.U = ctx[l]->U16;
                a.Ae = ctx[l]->A16[0];
                a.Aio = ctx[l]->Ai16[1];
            }
            return sap_operator<P>(ctx[l], *pl, a);
        };
        if (b->p == LQCD_F32)
            LQCD_TRY(again(std::integral_constant<int, LQCD_F32>()));
        else
            LQCD_TRY(again(std::integral_constant<int, LQCD_F16S>()));
    }
    return LQCD_OK;
}

// psi = M_sap eta on every lattice whose active flag is set (the arenas given
// at creation; eta: an arena of the same layout, bytes long)
lqcd_status sap_batch_apply(lqcd_ctx *hc, SapBatch *b, const void *eta, size_t bytes, const int *active)
{
    LQCD_CUDA_CHECK(hc, cudaMemsetAsync(b->psi, 0, bytes, hc->stream));
    LQCD_CUDA_CHECK(hc, cudaMemcpyAsync(b->r, eta, bytes, cudaMemcpyDeviceToDevice, hc->stream));
    LQCD_CUDA_CHECK(hc, cudaMemsetAsync(b->queue, 0, 2 * b->ncy * sizeof(int), hc->stream));
    return b->p == LQCD_F32 ? sap_batch_run<LQCD_F32>(hc, b, active) : sap_batch_run<LQCD_F16S>(hc, b, active);
}

void sap_free_plans(lqcd_ctx *c)
{
    for (auto it = g_plans.begin(); it != g_plans.end();) {
        if (it->ctx == c) {
            cudaFree(it->plan.blocks_dev);
            cudaFree(it->plan.face_dev[0]);
            cudaFree(it->plan.face_dev[1]);
            for (auto &pm : it->plan.perm) cudaFree(pm.p);
            it = g_plans.erase(it);
        } else
            ++it;
    }
}

extern "C" lqcd_status lqcd_sap(lqcd_ctx *c, const lqcd_sap_params *sp, const double *eta, double *psi)
{
    if (!c || !sp || !eta || !psi) return set_err(c, LQCD_ERR_ARG, "null argument");
    lqcd_prec p = sp->prec;
    if (p != LQCD_F64 && p != LQCD_F32 && p != LQCD_F16S) return set_err(c, LQCD_ERR_ARG, "SAP precision %d", (int)p);
    size_t fb = 2 * native_half_bytes(c, p);
    size_t fb64 = 2 * native_half_bytes(c, LQCD_F64);
    void *a, *b, *t;
    LQCD_TRY(ws_get(c, WS_SAP_IN, fb, &a));
    LQCD_TRY(ws_get(c, WS_SAP_PSI, fb, &b));
    LQCD_TRY(ws_get(c, WS_PACK_IN, fb64, &t));
    // canonical FP64 -> native FP64 -> native prec
    LQCD_TRY(pack_field(c, LQCD_F64, 2, eta, t, 1, false));
    LQCD_TRY(convert_native(c, LQCD_F64, p, t, a, 2));
    LQCD_TRY(sap_apply(c, sp, a, b));
    LQCD_TRY(convert_native(c, p, LQCD_F64, b, t, 2));
    return pack_field(c, LQCD_F64, 2, psi, t, 1, true);
}
