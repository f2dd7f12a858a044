// Wilson-clover stencil kernels on native (site-minor) layouts: the float
// single-field form and the dispatch of D, Dhat (Eq. 1, Eq. 2) over it, the
// register-blocked multi-field form (lqcd_dirac_mr.cu), the staged form
// (lqcd_dirac_sm.cu) and the FP64 form (lqcd_dirac_d.cu).
//
// One thread per (output site, right-hand side).  A CTA is blockDim.x sites
// by blockDim.y right-hand sides, so a warp reads 32 consecutive sites of one
// field (coalesced 16-byte loads) and the warps of the other right-hand
// sides reuse the same link / clover words from L1.
#include <type_traits>

#include "lqcd_stencil.cuh"
#include "lqcd_tune.h"

namespace {

using namespace stencil;

//   MODE_HOP  : out = -1/2 S
//   MODE_DHAT1: out = A^-1 (-1/2 S)            (chi_o = A_oo^-1 H_oe psi_e)
//   MODE_DHAT2: out = A in_same + 1/2 S        (A_ee psi_e - H_eo chi_o)
//   MODE_D    : out = A in_same - 1/2 S        (D psi on one parity)
// with S = sum of the 8 projected hops of in_other.
// occupancy variants: (max threads per CTA, min CTAs per SM)
template <int VAR>
struct Var;
template <>
struct Var<0> {
    static constexpr int T = 384, B = 1;
};
template <>
struct Var<1> {
    static constexpr int T = 384, B = 2;
};
template <>
struct Var<2> {
    static constexpr int T = 256, B = 3;
};
template <>
struct Var<3> {
    static constexpr int T = 256, B = 4;
};
constexpr int NVAR = 4;
inline int var_max_threads(int v) { return v < 2 ? 384 : 256; }

// output site r (rank of parity p_out), right-hand side k
template <class R, class SP, class LK, class CL, int MODE>
__device__ __forceinline__ void hop_site(const HopArgs<SP, LK, CL> &a, int r, int k)
{
    const long Vh = a.g.Vh;
    int x[4];
    rank_coords(a.g, a.p_out, r, x);
    const SP *in = a.in_other + k * a.in_rs;
    Spinor<R> acc;
    if (MODE == MODE_HOP || MODE == MODE_DHAT1) {
#pragma unroll
        for (int s = 0; s < 4; s++)
#pragma unroll
            for (int c = 0; c < 3; c++) acc.s[s][c] = mk(R(0), R(0));
    } else {
        // start from (1/f) A in_same, f = +-1/2 (exact power-of-two scaling), so the
        // hops accumulate into the same registers: out = f (A in / f + S)
        Spinor<R> self;
        load_spinor(a.in_same + k * a.same_rs, Vh, r, self);
        clover_apply<R, CL>(a.clov, Vh, r, self, acc);
        const R inv_f = MODE == MODE_DHAT2 ? R(2) : R(-2);
#pragma unroll
        for (int s = 0; s < 4; s++)
#pragma unroll
            for (int c = 0; c < 3; c++) acc.s[s][c] = inv_f * acc.s[s][c];
    }
    hop_dir<R, SP, LK, 0>(a.g, a.p_out, r, x, in, Vh, a.U, acc);
    hop_dir<R, SP, LK, 1>(a.g, a.p_out, r, x, in, Vh, a.U, acc);
    hop_dir<R, SP, LK, 2>(a.g, a.p_out, r, x, in, Vh, a.U, acc);
    hop_dir<R, SP, LK, 3>(a.g, a.p_out, r, x, in, Vh, a.U, acc);
    const R f = MODE == MODE_DHAT2 ? R(0.5) : R(-0.5);
#pragma unroll
    for (int s = 0; s < 4; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) acc.s[s][c] = f * acc.s[s][c];
    if (MODE == MODE_DHAT1) {
        Spinor<R> res;
        clover_apply<R, CL>(a.clov, Vh, r, acc, res);
        store_spinor(a.out + k * a.out_rs, Vh, r, res);
    } else {
        store_spinor(a.out + k * a.out_rs, Vh, r, acc);
    }
}

// one-dimensional grid: CTA b covers site tile b / ngy and field block b % ngy,
// so the CTAs of all fields of a site tile run next to each other and share
// its links and clover term through L1/L2
template <class R, class SP, class LK, class CL, int MODE, int VAR>
__global__ void __launch_bounds__(Var<VAR>::T, Var<VAR>::B) k_hop(const HopParam<MODE, SP, LK, CL> args, int ngy)
{
    after_previous();
    const HopArgs<SP, LK, CL> &a = hop_args<MODE>(args);
    const int gy = blockIdx.x % ngy, tile = blockIdx.x / ngy;
    const int r = tile * blockDim.x + threadIdx.x;
    const int k = gy * blockDim.y + threadIdx.y;
    if (r >= a.g.Vh || k >= a.nrhs) return;
    hop_site<R, SP, LK, CL, MODE>(a, r, k);
}

// One stage of Dhat (MODE_DHAT1, MODE_DHAT2) on several lattices in one launch.
// args[2 l + stage]: lattice l; items: (lattice, first rank of the tile, sites in
// the tile); tiles of lattices whose active flag is 0 are skipped.  shift moves
// the even input field.
template <class R, class SP, class LK, class CL, int MODE>
__global__ void __launch_bounds__(256) k_hop_batch(const HopArgs<SP, LK, CL> *args, const int4 *items, const int *active,
                                                   long shift)
{
    __shared__ HopArgs<SP, LK, CL> sa;
    const int4 w = items[blockIdx.x];
    if (active && !active[w.x]) return;
    if (threadIdx.x == 0) {
        sa = args[2 * w.x + (MODE == MODE_DHAT2)];
        if (MODE == MODE_DHAT1)
            sa.in_other += shift;
        else
            sa.in_same += shift;
    }
    __syncthreads();
    if ((int)threadIdx.x < w.z) hop_site<R, SP, LK, CL, MODE>(sa, w.y + threadIdx.x, 0);
}

template <class R, class SP, class LK, class CL, int MODE>
lqcd_status launch_var(lqcd_ctx *c, int var, dim3 b, const HopArgs2<SP, LK, CL> &a)
{
    const int ngy = div_up(a.nrhs, b.y);
    const long nb = (long)div_up(c->g.Vh, b.x) * ngy;
    if (nb > 0x7fffffffL) return set_err(c, LQCD_ERR_ARG, "stencil: grid of %ld CTAs", nb);
    const dim3 grid((unsigned)nb, hop_grid_y<MODE>());
    const bool pdl = c->hop_dep && !c->capturing;
    switch (var) {
        case 0: launch_pdl(pdl, k_hop<R, SP, LK, CL, MODE, 0>, grid, b, c->stream, a, ngy); break;
        case 1: launch_pdl(pdl, k_hop<R, SP, LK, CL, MODE, 1>, grid, b, c->stream, a, ngy); break;
        case 2: launch_pdl(pdl, k_hop<R, SP, LK, CL, MODE, 2>, grid, b, c->stream, a, ngy); break;
        default: launch_pdl(pdl, k_hop<R, SP, LK, CL, MODE, 3>, grid, b, c->stream, a, ngy); break;
    }
    c->n_kernel_launches++;
    LQCD_LAUNCH_CHECK(c);
    return LQCD_OK;
}

// candidate launch shapes: tx sites x ty fields per CTA
std::vector<TuneChoice> hop_candidates(int nrhs)
{
    std::vector<TuneChoice> v;
    std::vector<int> tys;
    for (int t : {nrhs, (nrhs + 1) / 2, (nrhs + 2) / 3, 4, 2, 1})
        if (t >= 1 && t <= nrhs && std::find(tys.begin(), tys.end(), t) == tys.end()) tys.push_back(t);
    for (int var = 0; var < NVAR; var++)
        for (int ty : tys)
            for (int tx : {16, 32, 64, 128, 256}) {
                int n = tx * ty;
                if (n > var_max_threads(var) || n < 64) continue;
                TuneChoice t;
                t.variant = var;
                t.tx = tx;
                t.ty = ty;
                v.push_back(t);
            }
    return v;
}

// LQCD_HOP_KIND = hop | mr | sm restricts the search to one kernel form
// (test instrumentation; ignored where that form does not exist, as in FP64),
// LQCD_HOP_KIND = d1 | d2 | d4 the FP64 search to one split G
int hop_force_split()
{
    const char *e = getenv("LQCD_HOP_KIND");
    return e && e[0] == 'd' && (e[1] == '1' || e[1] == '2' || e[1] == '4') && !e[2] ? e[1] - '0' : 0;
}
int hop_force_kind(bool has_alt, int nrhs)
{
    const char *e = getenv("LQCD_HOP_KIND");
    if (!e || !*e) return -1;
    const std::string k(e);
    if (k == "hop") return KIND_HOP;
    if (k == "mr" && has_alt && nrhs >= 2) return KIND_MR;
    if (k == "sm" && has_alt) return KIND_SM;
    return -1;
}

// staged shapes: tx sites (16 or 32) x ty fields per CTA
std::vector<TuneChoice> hop_sm_candidates(int nrhs)
{
    std::vector<TuneChoice> v;
    std::vector<int> tys;
    for (int t : {nrhs, (nrhs + 1) / 2, (nrhs + 2) / 3, 4, 2, 1})
        if (t >= 1 && t <= nrhs && std::find(tys.begin(), tys.end(), t) == tys.end()) tys.push_back(t);
    for (int var = 0; var < NVAR_SM; var++)
        for (int ty : tys)
            for (int tx : {16, 32}) {
                const int n = tx * ty;
                if (n > var_sm_max_threads(var) || n < 32) continue;
                TuneChoice t;
                t.kind = KIND_SM;
                t.variant = var;
                t.tx = tx;
                t.ty = ty;
                v.push_back(t);
            }
    return v;
}

// register-blocked shapes: nr fields per thread, tx sites x ty field groups
std::vector<TuneChoice> hop_mr_candidates(int nrhs)
{
    std::vector<TuneChoice> v;
    for (int nr : {2, 3}) {
        if (nr > nrhs) continue;
        const int groups = (nrhs + nr - 1) / nr;
        std::vector<int> tys;
        for (int t : {1, 2, (groups + 1) / 2, groups})
            if (t >= 1 && t <= groups && std::find(tys.begin(), tys.end(), t) == tys.end()) tys.push_back(t);
        for (int var = 0; var < NVAR_MR; var++)
            for (int ty : tys)
                for (int tx : {32, 64, 128, 256}) {
                    const int n = tx * ty;
                    if (n > var_mr_max_threads(var) || n < 64) continue;
                    TuneChoice t;
                    t.variant = var;
                    t.tx = tx;
                    t.ty = ty;
                    t.nr = nr;
                    t.kind = KIND_MR;
                    v.push_back(t);
                }
    }
    return v;
}

// FP64 splits: 2 G threads per site (nr = G)
std::vector<TuneChoice> hop_d_candidates(int only)
{
    std::vector<TuneChoice> v;
    for (int G : {1, 2, 4})
        if (only == 0 || only == G) {
            TuneChoice t;
            t.kind = KIND_D;
            t.nr = G;
            v.push_back(t);
        }
    return v;
}

template <class R, class SP, class LK, class CL, int MODE>
lqcd_status launch_choice(lqcd_ctx *c, const TuneChoice &t, const HopArgs2<SP, LK, CL> &a)
{
    if constexpr (std::is_same<R, float>::value && MODE != MODE_HOP) {
        if (t.kind == KIND_MR) return launch_hop_mr<R, SP, LK, CL, MODE>(c, t.nr, t.variant, dim3(t.tx, t.ty), a);
        if (t.kind == KIND_SM) return launch_hop_sm<R, SP, LK, CL, MODE>(c, t.variant, dim3(t.tx, t.ty), a);
    }
    if constexpr (std::is_same<R, double>::value)
        return launch_hop_d<MODE>(c, t.nr, a);
    else
        return launch_var<R, SP, LK, CL, MODE>(c, t.variant, dim3(t.tx, t.ty), a);
}

template <class R, class SP, class LK, class CL, int MODE>
lqcd_status launch_hop(lqcd_ctx *c, int p_out, const SP *in_other, long in_rs, const SP *in_same,
                       long same_rs, SP *out, long out_rs, const LK *U, const CL *clov, int nrhs,
                       const SP *in_other1 = nullptr, const SP *in_same1 = nullptr, SP *out1 = nullptr,
                       const CL *clov1 = nullptr)
{
    HopArgs2<SP, LK, CL> a;
    a.in_other1 = in_other1;
    a.in_same1 = in_same1;
    a.out1 = out1;
    a.clov1 = clov1;
    a.g = c->g;
    a.p_out = p_out;
    a.nrhs = nrhs;
    a.in_other = in_other;
    a.in_rs = in_rs;
    a.in_same = in_same;
    a.same_rs = same_rs;
    a.out = out;
    a.out_rs = out_rs;
    a.U = U;
    a.clov = clov;
    constexpr bool dbl = std::is_same<R, double>::value;
    const int prec = dbl ? 0 : (std::is_same<SP, h16s>::value ? 2 : 1);
    constexpr bool has_alt = std::is_same<R, float>::value && MODE != MODE_HOP;
    const int force = hop_force_kind(has_alt, nrhs);
    // MODE_D keys name the launch of both parities
    static const char *kname[2][4] = {{"k_hop4_hop", "k_hop4_mr", "k_hop4_sm", "k_hop4"},
                                      {"k_hop4x2_hop", "k_hop4x2_mr", "k_hop4x2_sm", "k_hop4x2"}};
    static const char *dname[2][5] = {{"k_hop_d", "k_hop_d1", "k_hop_d2", "", "k_hop_d4"},
                                      {"k_hop_dx2", "k_hop_d1x2", "k_hop_d2x2", "", "k_hop_d4x2"}};
    constexpr int both = MODE == MODE_D;
    const int split = dbl ? hop_force_split() : 0;
    TuneMemo &memo = c->tune[MODE][prec][p_out][nrhs % TUNE_SLOTS];
    const int forced = dbl ? 16 + split : force;
    TuneChoice tc;
    if (memo.gen == tune_generation() && memo.nrhs == nrhs && memo.force == forced) {
        tc.variant = memo.variant;
        tc.tx = memo.tx;
        tc.ty = memo.ty;
        tc.nr = memo.nr;
        tc.kind = memo.kind;
        return launch_choice<R, SP, LK, CL, MODE>(c, tc, a);
    }
    std::string key = tune_key(c, dbl ? dname[both][split] : kname[both][force >= 0 ? force : 3], MODE, prec, nrhs);
    bool settled = true;   // a choice of the table, not a default taken while the search is off
    if (!tune_lookup(key, &tc)) {
        tc = TuneChoice();
        tc.tx = nrhs == 1 ? 128 : 32;
        tc.ty = nrhs == 1 ? 1 : std::min(nrhs, 8);
        if (dbl) {
            // without timings: split until each of the 608 schedulers has two warps
            const long w = (long)c->g.Vh * nrhs / 16;
            tc.kind = KIND_D;
            tc.nr = split ? split : (w >= 1216 ? 1 : (w >= 608 ? 2 : 4));
        } else if (force == KIND_MR) {
            tc.kind = KIND_MR;
            tc.nr = 2;
            tc.tx = 64;
            tc.ty = 1;
        } else if (force == KIND_SM) {
            tc.kind = KIND_SM;
            tc.tx = 32;
            tc.ty = std::min(nrhs, 8);
        }
        if (tune_enabled()) {
            float best = 1e30f;
            std::vector<TuneChoice> cands;
            if (dbl)
                cands = hop_d_candidates(split);
            else if (force < 0 || force == KIND_HOP)
                cands = hop_candidates(nrhs);
            if (has_alt && (force < 0 || force == KIND_MR))
                for (const TuneChoice &m : hop_mr_candidates(nrhs)) cands.push_back(m);
            if (has_alt && (force < 0 || force == KIND_SM))
                for (const TuneChoice &m : hop_sm_candidates(nrhs)) cands.push_back(m);
            for (const TuneChoice &cand : cands) {
                float us;
                lqcd_status s = tune_time(c, [&]() { return launch_choice<R, SP, LK, CL, MODE>(c, cand, a); }, 3, &us);
                if (s != LQCD_OK) return s;
                if (tune_verbose())
                    fprintf(stderr, "tune %s: kind=%d nr=%d var=%d %dx%d %.1f us\n", key.c_str(), cand.kind, cand.nr,
                            cand.variant, cand.tx, cand.ty, us);
                if (us < best) {
                    best = us;
                    tc = cand;
                    tc.us = us;
                }
            }
            tune_store(key, tc);
        } else {
            settled = false;
        }
    }
    if (settled) memo = TuneMemo{tune_generation(), nrhs, forced, tc.variant, tc.tx, tc.ty, tc.nr, tc.kind};
    return launch_choice<R, SP, LK, CL, MODE>(c, tc, a);
}

}  // namespace

// Dependent launches (launch_pdl) are a choice for each operator, precision, number of
// fields and lattice.  They hide the set-up of a kernel's CTAs behind the kernel
// before; but the CTAs set up early go to the SMs that are through first, so a kernel
// of about one wave may have several CTAs on some SMs and none on others.  Plain /
// dependent, us an application in a run: FP64 Dhat, one field, 2048 even sites 20.5 / 15.3,
// 8192 45 / 60, 16384 82 / 78; F16S, three fields, 23520 even sites 20.5 / 25.2 or 15.4 by
// the kernels' forms.  So a run of applications is timed both ways once the forms are
// settled (0.3 ms to 15 ms on the first call); above DEP_LONG_US an application the
// difference is below 1 % and the launches are dependent.  Over 126 operators and sizes
// the choice is 1.2 % faster than dependent launches throughout, at most 17 % where
// those lost.
constexpr float DEP_LONG_US = 300.f;
constexpr float DEP_MARGIN = 1.05f;   // behind other kernels dependent launches still save their set-up
enum { OP_DHAT = 0, OP_D = 1 };
namespace {
template <class Run>
lqcd_status run_operator(lqcd_ctx *c, int op, lqcd_prec p, int nrhs, Run run)
{
    DepMemo &m = c->dep[op][p][nrhs % TUNE_SLOTS];
    c->hop_dep = true;
    if (m.gen == tune_generation() && m.nrhs == nrhs) {
        c->hop_dep = m.dep;
        return run();
    }
    const std::string key = tune_key(c, "k_hop_dep", op, (int)p, nrhs);
    TuneChoice t;
    if (!tune_lookup(key, &t)) {
        if (!tune_enabled()) return run();
        LQCD_TRY(run());   // settles the forms
        float us, best[2] = {1e30f, 1e30f};
        LQCD_TRY(tune_time(c, run, 1, &us));
        constexpr int N = 6;   // applications in a run
        for (int rep = 0; rep < 4 && us < DEP_LONG_US; rep++) {
            c->hop_dep = rep & 1;
            LQCD_TRY(tune_time(
                c,
                [&]() -> lqcd_status {
                    for (int i = 0; i < N; i++) LQCD_TRY(run());
                    return LQCD_OK;
                },
                1, &us));
            us /= N;
            if (tune_verbose()) fprintf(stderr, "tune %s: dependent=%d %.1f us\n", key.c_str(), rep & 1, us);
            best[rep & 1] = std::min(best[rep & 1], us);
        }
        t.variant = best[1] <= DEP_MARGIN * best[0];
        t.us = std::min(us, best[t.variant]);
        tune_store(key, t);
    }
    m = DepMemo{tune_generation(), nrhs, t.variant != 0};
    c->hop_dep = m.dep;
    return run();
}
template <class R, class SP, class LK, class CL>
lqcd_status launch_dhat(lqcd_ctx *c, lqcd_prec p, const void *in, long in_rs, void *out, long out_rs, void *tmp_o,
                        const LK *U, const CL *Aio, const CL *Ae, int nrhs)
{
    auto *i = (const SP *)in;
    auto *o = (SP *)out;
    auto *t = (SP *)tmp_o;
    const long rs = native_half_units(c, p);
    return run_operator(c, OP_DHAT, p, nrhs, [&]() -> lqcd_status {
        LQCD_TRY((launch_hop<R, SP, LK, CL, MODE_DHAT1>(c, 1, i, in_rs, nullptr, 0, t, rs, U, Aio, nrhs)));
        return launch_hop<R, SP, LK, CL, MODE_DHAT2>(c, 0, t, rs, i, in_rs, o, out_rs, U, Ae, nrhs);
    });
}
}  // namespace

// Dhat on native half fields: in / out even, in_rs / out_rs units apart per rhs
// (native units: double2, float4, h16s); tmp_o: nrhs odd half fields one after the other.
lqcd_status dirac_dhat_s(lqcd_ctx *c, lqcd_prec p, const void *in, long in_rs, void *out, long out_rs, void *tmp_o,
                         int nrhs)
{
    if (!c->have_clover) return set_err(c, LQCD_ERR_STATE, "clover term not built");
    if (p == LQCD_F64)
        return launch_dhat<double, double2, double2, double2>(c, p, in, in_rs, out, out_rs, tmp_o, c->U64, c->Ai64[1],
                                                              c->A64[0], nrhs);
    if (p == LQCD_F32)
        return launch_dhat<float, float4, float4, float4>(c, p, in, in_rs, out, out_rs, tmp_o, c->U32, c->Ai32[1],
                                                          c->A32[0], nrhs);
    if (p == LQCD_F16S)
        return launch_dhat<float, h16s, uint2, uint2>(c, p, in, in_rs, out, out_rs, tmp_o, c->U16, c->Ai16[1],
                                                      c->A16[0], nrhs);
    return set_err(c, LQCD_ERR_ARG, "precision %d not supported for Dhat", (int)p);
}
lqcd_status dirac_dhat(lqcd_ctx *c, lqcd_prec p, const void *in, void *out, void *tmp_o, int nrhs)
{
    const long rs = native_half_units(c, p);
    return dirac_dhat_s(c, p, in, rs, out, rs, tmp_o, nrhs);
}

// D on native full fields ([rhs][even half][odd half]), both parities in one
// launch: two launches of half the CTAs each left mid-size lattices with a partly
// filled wave (FP32, 28 x 12 x 10 x 14, 5 fields: two launches of 16.3 us -> 27.6 us).
namespace {
template <class R, class SP, class LK, class CL>
lqcd_status launch_D(lqcd_ctx *c, lqcd_prec p, const void *in, void *out, const LK *U, CL *const A[2], int nrhs)
{
    auto *i = (const SP *)in;
    auto *o = (SP *)out;
    const long h = native_half_units(c, p);
    return run_operator(c, OP_D, p, nrhs, [&]() {
        return launch_hop<R, SP, LK, CL, MODE_D>(c, 0, i + h, 2 * h, i, 2 * h, o, 2 * h, U, A[0], nrhs, i, i + h,
                                                 o + h, A[1]);
    });
}
}  // namespace

lqcd_status dirac_D(lqcd_ctx *c, lqcd_prec p, const void *in, void *out, int nrhs)
{
    if (!c->have_clover) return set_err(c, LQCD_ERR_STATE, "clover term not built");
    if (p == LQCD_F64) return launch_D<double, double2, double2, double2>(c, p, in, out, c->U64, c->A64, nrhs);
    if (p == LQCD_F32) return launch_D<float, float4, float4, float4>(c, p, in, out, c->U32, c->A32, nrhs);
    if (p == LQCD_F16S) return launch_D<float, h16s, uint2, uint2>(c, p, in, out, c->U16, c->A16, nrhs);
    return set_err(c, LQCD_ERR_ARG, "precision %d not supported for D", (int)p);
}

// out (parity p_out) = H in_other, native half fields with given rhs strides
lqcd_status dirac_hop_parity(lqcd_ctx *c, lqcd_prec p, int p_out, const void *in_other, void *out,
                             long in_rstride, long out_rstride, int nrhs)
{
    c->hop_dep = true;
    if (p == LQCD_F64)
        return launch_hop<double, double2, double2, double2, MODE_HOP>(
            c, p_out, (const double2 *)in_other, in_rstride, nullptr, 0, (double2 *)out, out_rstride,
            c->U64, (const double2 *)nullptr, nrhs);
    if (p == LQCD_F32)
        return launch_hop<float, float4, float4, float4, MODE_HOP>(
            c, p_out, (const float4 *)in_other, in_rstride, nullptr, 0, (float4 *)out, out_rstride,
            c->U32, (const float4 *)nullptr, nrhs);
    return set_err(c, LQCD_ERR_ARG, "precision %d not supported for hop", (int)p);
}

// ------------------------------------------------------------------ batches
struct DBatch {
    lqcd_prec p = LQCD_F32;
    int nlat = 0;
    long sites = 0;
    void *args = nullptr;                       // HopArgs[2 nlat]: (lattice, stage)
    int4 *items[3] = {nullptr, nullptr, nullptr};   // tiles of 64 / 128 / 256 ranks
    int nitems[3] = {0, 0, 0};
    int choice = -1;                            // tuned tile size index
};
static const int kBatchTile[3] = {64, 128, 256};

namespace {
template <class SP, class LK, class CL>
lqcd_status batch_args(lqcd_ctx *hc, DBatch *b, lqcd_ctx *const *ctx, int n, const SP *in, SP *tmp, SP *out,
                       const long *off, LK *lqcd_ctx::*U, CL *(lqcd_ctx::*A)[2], CL *(lqcd_ctx::*Ai)[2])
{
    std::vector<HopArgs<SP, LK, CL>> v;
    for (int l = 0; l < n; l++)
        for (int stage = 0; stage < 2; stage++) {
            HopArgs<SP, LK, CL> a = {};
            a.g = ctx[l]->g;
            a.p_out = 1 - stage;
            a.nrhs = 1;
            a.in_other = (stage == 0 ? in : tmp) + off[l];
            a.in_rs = 0;
            a.in_same = stage == 0 ? nullptr : in + off[l];
            a.same_rs = 0;
            a.out = (stage == 0 ? tmp : out) + off[l];
            a.out_rs = 0;
            a.U = ctx[l]->*U;
            a.clov = stage == 0 ? (ctx[l]->*Ai)[1] : (ctx[l]->*A)[0];
            v.push_back(a);
        }
    const size_t bytes = v.size() * sizeof(v[0]);
    if (cudaMalloc(&b->args, bytes) != cudaSuccess) {
        cudaGetLastError();
        return set_err(hc, LQCD_ERR_NOMEM, "batched Dhat arguments");
    }
    LQCD_CUDA_CHECK(hc, cudaMemcpy(b->args, v.data(), bytes, cudaMemcpyHostToDevice));
    return LQCD_OK;
}
}  // namespace

// in, tmp, out: arenas of half fields (even, odd, even), lattice l at off[l]
lqcd_status dirac_batch_create(lqcd_ctx *hc, lqcd_ctx *const *ctx, int n, lqcd_prec p, const void *in, void *tmp,
                               void *out, const long *off, DBatch **out_b)
{
    if (p != LQCD_F32 && p != LQCD_F64) return set_err(hc, LQCD_ERR_ARG, "batched Dhat: precision %d", (int)p);
    DBatch *b = new DBatch();
    b->p = p;
    b->nlat = n;
    lqcd_status st;
    if (p == LQCD_F32)
        st = batch_args<float4, float4, float4>(hc, b, ctx, n, (const float4 *)in, (float4 *)tmp, (float4 *)out, off,
                                                &lqcd_ctx::U32, &lqcd_ctx::A32, &lqcd_ctx::Ai32);
    else
        st = batch_args<double2, double2, double2>(hc, b, ctx, n, (const double2 *)in, (double2 *)tmp, (double2 *)out,
                                                   off, &lqcd_ctx::U64, &lqcd_ctx::A64, &lqcd_ctx::Ai64);
    for (int t = 0; t < 3 && st == LQCD_OK; t++) {
        std::vector<int4> it;
        for (int l = 0; l < n; l++)
            for (int r0 = 0; r0 < ctx[l]->g.Vh; r0 += kBatchTile[t])
                it.push_back(make_int4(l, r0, std::min(kBatchTile[t], ctx[l]->g.Vh - r0), 0));
        b->nitems[t] = (int)it.size();
        if (cudaMalloc(&b->items[t], it.size() * sizeof(int4)) != cudaSuccess) {
            cudaGetLastError();
            st = set_err(hc, LQCD_ERR_NOMEM, "batched Dhat work list");
        } else {
            cudaMemcpy(b->items[t], it.data(), it.size() * sizeof(int4), cudaMemcpyHostToDevice);
        }
    }
    if (st != LQCD_OK) {
        dirac_batch_free(b);
        return st;
    }
    for (int l = 0; l < n; l++) b->sites += ctx[l]->g.V;
    *out_b = b;
    return LQCD_OK;
}

void dirac_batch_free(DBatch *b)
{
    if (!b) return;
    cudaFree(b->args);
    for (int t = 0; t < 3; t++) cudaFree(b->items[t]);
    delete b;
}

namespace {
template <class R, class SP, class LK, class CL>
void batch_launch2(cudaStream_t st, const DBatch *b, int t, const int *active, long shift)
{
    auto *a = (const HopArgs<SP, LK, CL> *)b->args;
    k_hop_batch<R, SP, LK, CL, MODE_DHAT1><<<b->nitems[t], kBatchTile[t], 0, st>>>(a, b->items[t], active, shift);
    k_hop_batch<R, SP, LK, CL, MODE_DHAT2><<<b->nitems[t], kBatchTile[t], 0, st>>>(a, b->items[t], active, shift);
}
lqcd_status batch_launch(lqcd_ctx *hc, DBatch *b, int t, const int *active, long shift)
{
    if (b->p == LQCD_F32)
        batch_launch2<float, float4, float4, float4>(hc->stream, b, t, active, shift);
    else
        batch_launch2<double, double2, double2, double2>(hc->stream, b, t, active, shift);
    hc->n_kernel_launches += 2;
    LQCD_LAUNCH_CHECK(hc);
    return LQCD_OK;
}
}  // namespace

// out = Dhat (in + shift) on every lattice of the batch (tile size chosen by the
// autotuner on the first call, which must not be inside a stream capture)
lqcd_status dirac_batch_dhat(lqcd_ctx *hc, DBatch *b, long shift, const int *active)
{
    if (b->choice < 0) {
        std::string key = "k_hop_batch_dhat/p" + std::to_string((int)b->p) + "/n" + std::to_string(b->nlat) + "/s" +
                          std::to_string(b->sites);
        TuneChoice tc;
        if (tune_lookup(key, &tc)) {
            b->choice = tc.variant;
        } else {
            b->choice = 1;
            if (tune_enabled()) {
                float best = 1e30f;
                for (int t = 0; t < 3; t++) {
                    float us;
                    LQCD_TRY(tune_time(hc, [&]() { return batch_launch(hc, b, t, active, shift); }, 3, &us));
                    if (tune_verbose()) fprintf(stderr, "tune %s: tile %d %.1f us\n", key.c_str(), kBatchTile[t], us);
                    if (us < best) {
                        best = us;
                        b->choice = t;
                    }
                }
                tc.variant = b->choice;
                tc.tx = kBatchTile[b->choice];
                tc.us = best;
                tune_store(key, tc);
            }
        }
    }
    return batch_launch(hc, b, b->choice, active, shift);
}
