// FP64 stencil with a site's work split over 2 G threads (G = 1, 2, 4).
//
// What bounds it is GB300's FP64 pipe: about 1160 multiply-adds per site and
// field against 2 per clock and SM, so a thread that owns a whole site runs for
// about 40 us however small the lattice is, and holds 200 registers.  The
// split follows the spin structure.  Thread s = 0, 1 takes component s of every
// half spinor h = psi_up -+ e_mu psi_lo: e_mu maps the lower spin s (mu = 0, 3)
// or 1 - s (mu = 1, 2) onto it, so the thread multiplies one colour vector per
// hop and adds to one upper and one lower spin, and nothing is computed twice.
// Those two kinds k of directions are the next split (G = 2), the two senses
// of a direction the last (G = 4; the two threads exchange their products and
// one sums the upper spin, the other the lower).  The sums of the kinds meet by
// lane shuffles and the rows of the clover block are shared out in the same way.
//
// Every form adds in one order -- per kind the forward hops of its two
// directions, then the backward ones, then the two kinds -- so results do not
// depend on G and the autotuner may choose.  CTAs of 32, 64 and 128 threads and
// occupancies of 3 and 5 CTAs were timed and differ by less than 1 %.
// Measured per launch, one field: 8^4 40 us (a thread per site) -> 8.0 us (G = 4;
// 15 for G = 2, 24 for G = 1), 48 x 24^3 695 -> 660 us (G = 1, 90 % of the FP64
// pipe; G = 2 670, G = 4 730).
#include "lqcd_stencil.cuh"

namespace stencil {

namespace {

constexpr int HOP_D_THREADS = 128;

struct HopSite {
    int x[4], lex;
    unsigned keep;   // bit 2 mu + fwd: the hop stays in the site's block
};

__device__ __forceinline__ double shx(double v, int m) { return __shfl_xor_sync(0xffffffffu, v, m); }
__device__ __forceinline__ void shx3(const cx<double> v[3], int m, cx<double> o[3])
{
#pragma unroll
    for (int c = 0; c < 3; c++) o[c] = mk(shx(v[c].re, m), shx(v[c].im, m));
}

// v with its sign bit xored: unlike -v, never an operation of the FP64 pipe
__device__ __forceinline__ double flip(unsigned mask, double v)
{
    return __hiloint2double(__double2hiint(v) ^ (int)mask, __double2loint(v));
}
__device__ __forceinline__ unsigned sign_mask(bool neg) { return neg ? 0x80000000u : 0u; }

// Product of the hop of direction mu in the given sense, spin component s:
// w = s_bc U h or s_bc U^dag h, s_bc the time-boundary sign.  Signs, factors i
// and (SENSE = 0: fwd at run time; +1, -1: fixed) the adjoint are selected on
// the integer side: the FP64 pipe sees 6 + 36 operations.
// BLK: a hop out of the site's block gives w = 0 (and no work where no lane of
// the warp keeps its hop).
template <int SENSE, bool BLK>
__device__ __forceinline__ void hop_w(const Geom &g, int p_out, int r, const HopSite &S, int mu, bool fwd_rt, int s,
                                      const double2 *__restrict__ in, const double2 *__restrict__ U, cx<double> w[3])
{
    const bool fwd = SENSE == 0 ? fwd_rt : SENSE > 0;
    const long Vh = g.Vh;
    const bool keep = !BLK || (S.keep >> (2 * mu + fwd) & 1);
    if (BLK && !__any_sync(0xffffffffu, keep)) {
#pragma unroll
        for (int c = 0; c < 3; c++) w[c] = mk(0.0, 0.0);
        return;
    }
    const bool swap = mu == 1 || mu == 2, imag = mu & 1;
    const int xm = mu == 0 ? S.x[0] : (mu == 1 ? S.x[1] : (mu == 2 ? S.x[2] : S.x[3]));
    const int Lm = mu == 0 ? g.L[0] : (mu == 1 ? g.L[1] : (mu == 2 ? g.L[2] : g.L[3]));
    const int st = mu == 3 ? 1 : (mu == 2 ? g.L[3] : (mu == 1 ? g.L[2] * g.L[3] : g.L[1] * g.L[2] * g.L[3]));
    const bool edge = xm == (fwd ? Lm - 1 : 0);
    const int step = edge ? -(Lm - 1) * st : st;
    const int n = (S.lex + (fwd ? step : -step)) >> 1;
    const double2 *pu = in + 3L * s * Vh + n;
    const double2 *pl = in + (6L + 3 * (swap ? 1 - s : s)) * Vh + n;
    const double2 *ul = U + (long)(((fwd ? p_out : 1 - p_out) * 4 + mu) * 9) * Vh + (fwd ? r : n);
    double2 a[3], b[3], u[9];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        a[c] = __ldg(pu + c * Vh);
        b[c] = __ldg(pl + c * Vh);
    }
#pragma unroll
    for (int e = 0; e < 9; e++) u[e] = __ldg(ul + e * Vh);
    // e_mu psi_lo = es (l or i l), es = +1 only for s = 1 and mu = 2, 3; h = psi_up -+ e_mu psi_lo
    const unsigned neg = sign_mask(fwd == (mu >= 2 && s)), negi = neg ^ sign_mask(imag);
    cx<double> h[3], m[3][3];
#pragma unroll
    for (int c = 0; c < 3; c++)
        h[c] = mk(a[c].x + flip(negi, imag ? b[c].y : b[c].x), a[c].y + flip(neg, imag ? b[c].x : b[c].y));
    const unsigned conj = sign_mask(!fwd);
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const double2 f = u[3 * i + j], d = u[3 * j + i];
            if (SENSE == 0)
                m[i][j] = mk(fwd ? f.x : d.x, flip(conj, fwd ? f.y : d.y));
            else
                m[i][j] = mk(f.x, f.y);
        }
    if (SENSE >= 0)
        su3_vec(m, h, w);
    else
        su3dag_vec(m, h, w);
    const unsigned bc = sign_mask(mu == 0 && edge && g.bc_t < 0);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        w[c] = mk(flip(bc, w[c].re), flip(bc, w[c].im));
        if (BLK && !keep) w[c] = mk(0.0, 0.0);
    }
}

// what w adds to the lower spin: sgn e_mu^dag w
__device__ __forceinline__ void lower_of(int mu, bool fwd, int s, const cx<double> w[3], cx<double> l[3])
{
    const bool imag = mu & 1;
    const unsigned neg = sign_mask(fwd == (mu >= 2 && s)), negi = neg ^ sign_mask(imag);
#pragma unroll
    for (int c = 0; c < 3; c++)
        l[c] = mk(flip(neg, imag ? w[c].im : w[c].re), flip(negi, imag ? w[c].re : w[c].im));
}

__device__ __forceinline__ void add3(cx<double> a[3], const cx<double> b[3])
{
#pragma unroll
    for (int c = 0; c < 3; c++) a[c] = a[c] + b[c];
}

// the four hops of kind k (directions ma, mb), forward first
template <bool BLK>
__device__ __forceinline__ void hop_kind(const Geom &g, int p_out, int r, const HopSite &S, int ma, int mb, int s,
                                         const double2 *__restrict__ in, const double2 *__restrict__ U,
                                         cx<double> up[3], cx<double> lo[3])
{
    cx<double> w[3], l[3];
    hop_w<1, BLK>(g, p_out, r, S, ma, true, s, in, U, up);
    lower_of(ma, true, s, up, lo);
    auto more = [&](int mu, bool fwd) {
        add3(up, w);
        lower_of(mu, fwd, s, w, l);
        add3(lo, l);
    };
    hop_w<1, BLK>(g, p_out, r, S, mb, true, s, in, U, w);
    more(mb, true);
    hop_w<-1, BLK>(g, p_out, r, S, ma, false, s, in, U, w);
    more(ma, false);
    hop_w<-1, BLK>(g, p_out, r, S, mb, false, s, in, U, w);
    more(mb, false);
}

// row c of spin s (0, 1) of the packed Hermitian block blk at rank r, times the
// block vector: own0..own2 = components c, c + 1, c + 2 (mod 3) of spin s, oth =
// spin 1 - s.  c and s may differ between the lanes.
__device__ __forceinline__ cx<double> herm_row(const double2 *__restrict__ A, long Vh, int r, int blk, int s, int c,
                                               cx<double> own0, cx<double> own1, cx<double> own2,
                                               const cx<double> oth[3])
{
    const double2 *b = A + 18L * blk * Vh + r;
    const int i = 3 * s + c;
    const double2 dd = __ldg(b + (i >> 1) * Vh);
    const double d = (i & 1) ? dd.y : dd.x;
    cx<double> t = mk(d * own0.re, d * own0.im);
    auto off = [](int lo, int hi) { return 3 + lo * 5 - (lo * (lo - 1)) / 2 + (hi - lo - 1); };   // slot of (lo, hi)
    auto acc = [&](double2 o, bool conj, cx<double> v) {
        const double im = flip(sign_mask(conj), o.y);
        t.re = fmx(o.x, v.re, t.re);
        t.re = fmx(-im, v.im, t.re);
        t.im = fmx(o.x, v.im, t.im);
        t.im = fmx(im, v.re, t.im);
    };
    const int c1 = c == 2 ? 0 : c + 1, c2 = c == 0 ? 2 : c - 1;
    acc(__ldg(b + off(3 * s + min(c, c1), 3 * s + max(c, c1)) * Vh), c1 < c, own1);
    acc(__ldg(b + off(3 * s + min(c, c2), 3 * s + max(c, c2)) * Vh), c2 < c, own2);
#pragma unroll
    for (int j = 0; j < 3; j++) acc(__ldg(b + off(s ? j : c, s ? 3 + c : 3 + j) * Vh), s != 0, oth[j]);
    return t;
}

// Modes as in k_hop.  Lane = part * (32 / P) + site, P = 2 G parts per site:
// part bit 0 is s, bit 1 (G >= 2) the kind k, bit 2 (G = 4) the sense.
// One-dimensional grid, the fields of a site tile next to each other.
// BLK: the Dirichlet operator of blocks of extents bs.
struct BlkExt {
    int bs[4];
};
template <int MODE, int G, bool BLK = false>
__global__ void __launch_bounds__(HOP_D_THREADS, 3) k_hop_d(const HopParam<MODE, double2, double2, double2> args,
                                                            BlkExt bx)
{
    constexpr int P = 2 * G, SW = 32 / P;
    after_previous();
    const HopArgs<double2, double2, double2> &a = hop_args<MODE>(args);
    const long Vh = a.g.Vh;
    const int kf = blockIdx.x % a.nrhs;
    const int lane = threadIdx.x & 31, part = lane / SW, s = part & 1;
    const int tile = blockIdx.x / a.nrhs;
    const int r0 = (tile * (blockDim.x >> 5) + (threadIdx.x >> 5)) * SW + lane % SW;
    const bool ok = r0 < a.g.Vh;
    const int r = ok ? r0 : a.g.Vh - 1;   // every lane takes part in the shuffles
    HopSite S;
    rank_coords(a.g, a.p_out, r, S.x);
    S.lex = S.x[3] + a.g.L[3] * (S.x[2] + a.g.L[2] * (S.x[1] + a.g.L[1] * S.x[0]));
    if (BLK) {
        S.keep = 0;
#pragma unroll
        for (int m = 0; m < 4; m++) {
            const int L = a.g.L[m], b = bx.bs[m], l = S.x[m] % b;
            // a block that spans the direction keeps its wrapped hop
            S.keep |= (unsigned)(l + 1 < b || b == L) << (2 * m + 1) | (unsigned)(l > 0 || b == L) << (2 * m);
        }
    }
    const double2 *in = a.in_other + kf * a.in_rs;
    // sums of the hops: up of spin s, lo of the lower spin reached from it; for
    // G = 4 the thread keeps one of the two (up for sense bit 0, lo for 1) in up
    cx<double> up[3], lo[3];
    const int k0 = G >= 2 ? (part >> 1) & 1 : 0, d0 = G == 4 ? part >> 2 : 0;
    const int ma = k0 ? 1 : 0, mb = k0 ? 2 : 3;
    int sl = s;   // the lower spin that lo ends on
    if (G == 4) {
        cx<double> wa[3], wb[3], oa[3], ob[3], l[3];
        hop_w<0, BLK>(a.g, a.p_out, r, S, ma, d0 == 0, s, in, a.U, wa);
        hop_w<0, BLK>(a.g, a.p_out, r, S, mb, d0 == 0, s, in, a.U, wb);
        shx3(wa, 4 * SW, oa);
        shx3(wb, 4 * SW, ob);
        auto pick = [&](int mu, bool fwd, const cx<double> mine[3], const cx<double> other[3], cx<double> o[3]) {
            cx<double> w[3];
#pragma unroll
            for (int c = 0; c < 3; c++) w[c] = fwd == (d0 == 0) ? mine[c] : other[c];
            lower_of(mu, fwd, s, w, l);
#pragma unroll
            for (int c = 0; c < 3; c++) o[c] = d0 ? l[c] : w[c];
        };
        cx<double> t[3];
        pick(ma, true, wa, oa, up);
        pick(mb, true, wb, ob, t);
        add3(up, t);
        pick(ma, false, wa, oa, t);
        add3(up, t);
        pick(mb, false, wb, ob, t);
        add3(up, t);
        // the other kind: upper spin s in thread s, lower spin in thread 1 - s
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const int from = (d0 ? 3 : 2) * SW;
            const int src = (threadIdx.x & 31) ^ from;
            t[c] = mk(__shfl_sync(0xffffffffu, up[c].re, src), __shfl_sync(0xffffffffu, up[c].im, src));
        }
        add3(up, t);
        sl = k0 ? 1 - s : s;
    } else {
        hop_kind<BLK>(a.g, a.p_out, r, S, ma, mb, s, in, a.U, up, lo);
        cx<double> t[3];
        if (G == 1) {
            cx<double> u1[3], l1[3];
            hop_kind<BLK>(a.g, a.p_out, r, S, 1, 2, s, in, a.U, u1, l1);
            add3(up, u1);
            shx3(l1, SW, t);   // kind 1 of thread 1 - s ends on lower spin s
            add3(lo, t);
        } else {
            shx3(up, 2 * SW, t);
            add3(up, t);
            shx3(lo, 3 * SW, t);
            add3(lo, t);
            sl = k0 ? 1 - s : s;
        }
    }
    const double f = MODE == MODE_DHAT2 ? 0.5 : -0.5;
    double2 *out = a.out + kf * a.out_rs + r;
    auto put = [&](int spin, int c, cx<double> v) {
        if (ok) out[(3L * spin + c) * Vh] = make_double2(v.re, v.im);
    };
    if constexpr (MODE == MODE_HOP) {
#pragma unroll
        for (int c = 0; c < 3; c++) {
            if (G == 1 || (G == 2 && k0 == 0)) put(s, c, f * up[c]);
            if (G == 1 || (G == 2 && k0 == 1)) put(2 + sl, c, f * lo[c]);
            if (G == 4 && k0 == 0) put(d0 ? 2 + sl : s, c, f * up[c]);
        }
    } else {
        // G = 1: the thread's rows are spin s of both chirality blocks; G = 2: spin s
        // of the upper block (k0 = 0) or spin sl of the lower one; G = 4: the block
        // goes by d0, its rows 0, 1 and 2 to the two kinds
#pragma unroll
        for (int half = 0; half < (G == 1 ? 2 : 1); half++) {
            const int blk = G == 1 ? half : (G == 2 ? k0 : d0);
            const int sp = blk ? sl : s;
            cx<double> sum[3], own[3], oth[3];
#pragma unroll
            for (int c = 0; c < 3; c++) sum[c] = G != 4 && blk ? lo[c] : up[c];
            if (MODE == MODE_DHAT1) {
#pragma unroll
                for (int c = 0; c < 3; c++) own[c] = f * sum[c];
                shx3(own, SW, oth);
            } else {
                const double2 *same = a.in_same + kf * a.same_rs + r;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const double2 v = __ldg(same + (6L * blk + 3 * sp + c) * Vh);
                    const double2 w = __ldg(same + (6L * blk + 3 * (1 - sp) + c) * Vh);
                    own[c] = mk(v.x, v.y);
                    oth[c] = mk(w.x, w.y);
                }
            }
            auto row = [&](int c, cx<double> o0, cx<double> o1, cx<double> o2, cx<double> sm) {
                cx<double> t = herm_row(a.clov, Vh, r, blk, sp, c, o0, o1, o2, oth);
                if (MODE != MODE_DHAT1) t = mk(fmx(f, sm.re, t.re), fmx(f, sm.im, t.im));
                put(2 * blk + sp, c, t);
            };
            if (G == 4) {
                const bool z = k0;
                row(z ? 2 : 0, z ? own[2] : own[0], z ? own[0] : own[1], z ? own[1] : own[2], z ? sum[2] : sum[0]);
                if (!z) row(1, own[1], own[2], own[0], sum[1]);
            } else {
#pragma unroll
                for (int c = 0; c < 3; c++) row(c, own[c], own[(c + 1) % 3], own[(c + 2) % 3], sum[c]);
            }
        }
    }
}

}  // namespace

namespace {
template <int MODE, bool BLK>
lqcd_status launch_d(lqcd_ctx *c, int G, const HopArgs2<double2, double2, double2> &a, BlkExt bx)
{
    const int sites = HOP_D_THREADS / (2 * G);   // per CTA
    const long nb = (long)div_up(c->g.Vh, sites) * a.nrhs;
    if (nb > 0x7fffffffL) return set_err(c, LQCD_ERR_ARG, "FP64 stencil: grid of %ld CTAs", nb);
    const dim3 grid((unsigned)nb, hop_grid_y<MODE>());
    const bool pdl = c->hop_dep && !c->capturing;
    switch (G) {
        case 1: launch_pdl(pdl, k_hop_d<MODE, 1, BLK>, grid, HOP_D_THREADS, c->stream, a, bx); break;
        case 2: launch_pdl(pdl, k_hop_d<MODE, 2, BLK>, grid, HOP_D_THREADS, c->stream, a, bx); break;
        case 4: launch_pdl(pdl, k_hop_d<MODE, 4, BLK>, grid, HOP_D_THREADS, c->stream, a, bx); break;
        default: return set_err(c, LQCD_ERR_ARG, "FP64 stencil: split %d", G);
    }
    c->n_kernel_launches++;
    LQCD_LAUNCH_CHECK(c);
    return LQCD_OK;
}
}  // namespace

template <int MODE>
lqcd_status launch_hop_d(lqcd_ctx *c, int G, const HopArgs2<double2, double2, double2> &a)
{
    return launch_d<MODE, false>(c, G, a, BlkExt{});
}

lqcd_status launch_dhat_block_d(lqcd_ctx *c, const int bs[4], const double2 *in, double2 *tmp, double2 *out)
{
    HopArgs2<double2, double2, double2> a = {};
    a.g = c->g;
    a.nrhs = 1;
    a.in_rs = a.same_rs = a.out_rs = 0;
    a.U = c->U64;
    const BlkExt bx = {{bs[0], bs[1], bs[2], bs[3]}};
    c->hop_dep = true;
    // as the untuned rule of the lattice-wide operator
    const int G = c->g.Vh >= 16 * 1216 ? 1 : (c->g.Vh >= 16 * 608 ? 2 : 4);
    a.p_out = 1;
    a.in_other = in;
    a.in_same = nullptr;
    a.out = tmp;
    a.clov = c->Ai64[1];
    LQCD_TRY((launch_d<MODE_DHAT1, true>(c, G, a, bx)));
    a.p_out = 0;
    a.in_other = tmp;
    a.in_same = in;
    a.out = out;
    a.clov = c->A64[0];
    return launch_d<MODE_DHAT2, true>(c, G, a, bx);
}

template lqcd_status launch_hop_d<MODE_HOP>(lqcd_ctx *, int, const HopArgs2<double2, double2, double2> &);
template lqcd_status launch_hop_d<MODE_DHAT1>(lqcd_ctx *, int, const HopArgs2<double2, double2, double2> &);
template lqcd_status launch_hop_d<MODE_DHAT2>(lqcd_ctx *, int, const HopArgs2<double2, double2, double2> &);
template lqcd_status launch_hop_d<MODE_D>(lqcd_ctx *, int, const HopArgs2<double2, double2, double2> &);

}  // namespace stencil
