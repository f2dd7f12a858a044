// Outer solvers: the flexible GCR of Sec. 3-4, preconditioned by SAP or deflated
// SAP, and the solver entry points (CGNR: lqcd_cgnr.cu).
//
// The GCR solves either D psi = eta on the full lattice or Dhat psi_e = eta_e.
// The latter is the former with the odd half eliminated: completing an even
// field x_e by x_o = -A_oo^-1 H_oe x_e gives D x = (Dhat x_e, 0), so with a
// residual (rho_e, 0) the preconditioner M of the full lattice is applied as it
// is, the even half of its output is the search direction, and D phi_k needs
// Dhat phi_e alone (as many hops as D).  Every Krylov vector, dot product and
// update has half the length, and the residual is that of the Dhat system
// itself (Eq. 5 only bounds it by the full one, so that the full-lattice form went
// on with a tighter tolerance where needed).  Iteration counts are the same or
// lower: 62 at 32 x 16^3, one source, FP32 SAP, FP64 Krylov vectors, 70.9 -> 58.4 ms; 27 ->
// 26 at 48 x 24^3, 12 sources, deflated, build included 1218 -> 1101 ms.
//
// Precision: the residual, the solution update and the restart residual
// eta - D psi are FP64.  The preconditioner and D phi_k may run in FP32
// ("inner" precision), and with krylov = F32 the Krylov vectors and their
// Gram-Schmidt are FP32 too (FP64 sums); the recursive residual then carries
// FP32-level errors, so a cycle stops once it has gained ~1e-5 and the next
// cycle restarts from the FP64 true residual.
#include <chrono>
#include <cmath>
#include <vector>

#include "lqcd_internal.cuh"

namespace {

double now_s()
{
    return std::chrono::duration<double>(std::chrono::steady_clock::now().time_since_epoch()).count();
}

struct Cplx {
    double re, im;
};
inline Cplx cmul(Cplx a, Cplx b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
inline Cplx cdiv(Cplx a, double b) { return {a.re / b, a.im / b}; }

// ---------------------------------------------------------------- GCR
// All fields below are native full FP64 fields; nrhs of them are stored one
// after the other (stride nf double2).  The GCR of every right-hand side runs
// in lockstep so that the preconditioner, D and the BLAS-1 kernels each cover
// the whole batch in one launch; every right-hand side keeps its own
// Gram-Schmidt coefficients, and a converged one receives zero updates.

// phi = M rho
lqcd_status precond(lqcd_ctx *c, const lqcd_solver_params *sp, const double2 *rho, double2 *phi, int nrhs)
{
    const lqcd_sap_params &sap = sp->sap;
    if (sp->solver == LQCD_SOLVER_DFL_SAP_GCR) return dfl_precond_native(c, &sap, rho, phi, nrhs);
    if (sp->solver == LQCD_SOLVER_NET_GCR) return net_apply_native(c, rho, phi, nrhs);
    if (sp->solver == LQCD_SOLVER_DFL_NET_GCR) return dfl_precond_native(c, &sap, rho, phi, nrhs, true);
    if (sap.prec == LQCD_F64) return sap_apply(c, &sap, rho, phi, nrhs);
    void *a, *b;
    size_t fb = 2 * native_half_bytes(c, sap.prec) * nrhs;
    LQCD_TRY(ws_get(c, WS_SAP_IN, fb, &a));
    LQCD_TRY(ws_get(c, WS_SAP_PSI, fb, &b));
    LQCD_TRY(convert_native(c, LQCD_F64, sap.prec, rho, a, 2 * nrhs));
    LQCD_TRY(sap_apply(c, &sap, a, b, nrhs));
    return convert_native(c, sap.prec, LQCD_F64, b, phi, 2 * nrhs);
}

// chi = D phi (nh = 2) or Dhat phi_e (nh = 1) in the inner precision, phi nrhs
// native full FP64 fields, chi nrhs fields of nh halves
lqcd_status apply_D_inner(lqcd_ctx *c, lqcd_prec inner, int nh, const double2 *phi, double2 *chi, int nrhs)
{
    const long Vh = c->g.Vh;
    if (inner == LQCD_F64 && nh == 2) return dirac_D(c, LQCD_F64, phi, chi, nrhs);
    const size_t hb = native_half_bytes(c, inner);
    void *t = nullptr;
    if (nh == 1) LQCD_TRY(ws_get(c, WS_TMP_O, hb * nrhs, &t));
    if (inner == LQCD_F64) return dirac_dhat_s(c, LQCD_F64, phi, 24 * Vh, chi, 12 * Vh, t, nrhs);
    void *a, *b;
    const size_t fb = nh * hb * nrhs;
    LQCD_TRY(ws_get(c, WS_MISC, fb, &a));
    LQCD_TRY(ws_get(c, WS_MISC2, fb, &b));
    if (nh == 2) {
        LQCD_TRY(convert_native(c, LQCD_F64, inner, phi, a, 2 * nrhs));
        LQCD_TRY(dirac_D(c, inner, a, b, nrhs));
    } else {
        LQCD_TRY(convert_native(c, LQCD_F64, inner, phi, a, nrhs, 2, 1));
        LQCD_TRY(dirac_dhat(c, inner, a, b, t, nrhs));
    }
    return convert_native(c, inner, LQCD_F64, b, chi, nh * nrhs);
}

struct GcrState {
    std::vector<int> iters, restarts, net_fallbacks;
    std::vector<double> relres;
    std::vector<lqcd_status> status;
    explicit GcrState(int nrhs)
        : iters(nrhs, 0), restarts(nrhs, 0), net_fallbacks(nrhs, 0), relres(nrhs, 0),
          status(nrhs, LQCD_ERR_NOT_CONVERGED)
    {
    }
};

// LQCD_PROFILE=1: synchronise around the phases of the GCR and report their
// wall time on stderr (developer instrumentation; off by default)
struct PhaseProf {
    bool on;
    double t[4] = {0, 0, 0, 0};
    double t0 = 0;
    explicit PhaseProf(lqcd_ctx *c) : on(getenv("LQCD_PROFILE") && getenv("LQCD_PROFILE")[0] == '1'), ctx(c) {}
    lqcd_ctx *ctx;
    void start()
    {
        if (!on) return;
        cudaStreamSynchronize(ctx->stream);
        t0 = now_s();
    }
    void stop(int i)
    {
        if (!on) return;
        cudaStreamSynchronize(ctx->stream);
        t[i] += now_s() - t0;
    }
    ~PhaseProf()
    {
        if (!on) return;
        fprintf(stderr, "[lqcd gcr] precond %.4f s, D_inner %.4f s, gram-schmidt %.4f s, restart %.4f s\n", t[0],
                t[1], t[2], t[3]);
        double *p = ctx->prof_t;
        if (p[0] + p[1] + p[2] + p[3] + p[4] + p[5] > 0)
            fprintf(stderr,
                    "[lqcd dfl] project %.4f s, coarse %.4f s, expand %.4f s, D+sub %.4f s, sap %.4f s, "
                    "axpy %.4f s\n",
                    p[0], p[1], p[2], p[3], p[4], p[5]);
        fprintf(stderr, "[lqcd gcr] gram-schmidt %.1f GB, %.0f GB/s, %ld second passes\n", ctx->prof_gs_bytes * 1e-9,
                t[2] > 0 ? ctx->prof_gs_bytes * 1e-9 / t[2] : 0.0, ctx->prof_gs_second);
        for (int i = 0; i < 8; i++) p[i] = 0;
        ctx->prof_gs_bytes = 0;
        ctx->prof_gs_second = 0;
    }
};

// Krylov-vector storage of the GCR.  Krylov64: phi_k and chi_k native F64
// fields.  Krylov32 (krylov = inner = F32): phi_k and chi_k native F32 fields,
// so D phi_k runs on them directly and the Gram-Schmidt moves half the bytes
// and leaves GB300's FP64 pipe (FP64 products bound it at about a third of HBM
// bandwidth); rho and psi stay F64, the products with FP32 vectors are formed
// in float and accumulated in double.
//
// nh: halves per vector (1: the Dhat system).  phi_k and rho are full fields in
// either case (fphi, 24 Vh apart): the preconditioner writes and reads them, the
// odd half of rho being zero when nh = 1; chi, psi and eta have nh halves.
struct Krylov64 {
    using T = double2;
    lqcd_ctx *c;
    const lqcd_solver_params *sp;
    int nh, nrhs;
    long fphi, fchi, frho;   // elements between right-hand sides
    Krylov64(lqcd_ctx *ctx, const lqcd_solver_params *p, int halves, int n)
        : c(ctx), sp(p), nh(halves), nrhs(n), fphi(24 * (long)ctx->g.Vh), fchi(12L * halves * ctx->g.Vh),
          frho(24 * (long)ctx->g.Vh)
    {
    }
    lqcd_status precond_with(const lqcd_solver_params *p, const double2 *rho, T *ph)
    {
        return precond(c, p, rho, ph, nrhs);
    }
    lqcd_status D_inner(const T *ph, T *ch) { return apply_D_inner(c, sp->inner, nh, ph, ch, nrhs); }
    lqcd_status dots(const T *A, const T *B, int kk, double *out)
    {
        return bblas_dot(c, 2 * fchi, nrhs, (const double *)A, 2 * nrhs * fchi, 2 * fchi, (const double *)B, 2 * fchi,
                         kk, out);
    }
    lqcd_status axpy(int k, const double *cf, const T *X, T *y, double sign)
    {
        return bblas_multi_axpy(c, 2 * fchi, nrhs, k, cf, (const double *)X, 2 * nrhs * fchi, 2 * fchi, (double *)y,
                                2 * fchi, sign);
    }
    // |chi|^2 and <rho, chi>
    lqcd_status norm_rdot(const T *ch, const double2 *rho, double *out)
    {
        return bnorm_rdot64(c, nh, nrhs, ch, fchi, rho, frho, out);
    }
    // rho -= cR chi; chi *= s
    lqcd_status rho_update(const double *cR, const double *s, T *ch, double2 *rho)
    {
        return brho_update64(c, nh, nrhs, cR, s, ch, fchi, rho, frho);
    }
    lqcd_status psi_update(int nk, const double *cf, const T *phi, double2 *psi)
    {
        return bblas_multi_axpy(c, 2 * fchi, nrhs, nk, cf, (const double *)phi, 2 * nrhs * fphi, 2 * fphi,
                                (double *)psi, 2 * fchi, 1.0);
    }
    double final_fields() const { return 5.0; }   // F64-field transfers of norm_rdot + rho_update
};

struct Krylov32 {
    using T = float4;
    lqcd_ctx *c;
    const lqcd_solver_params *sp;
    int nh, nrhs;
    long fphi, fchi, frho;   // elements between right-hand sides
    Krylov32(lqcd_ctx *ctx, const lqcd_solver_params *p, int halves, int n)
        : c(ctx), sp(p), nh(halves), nrhs(n), fphi(12 * (long)ctx->g.Vh), fchi(6L * halves * ctx->g.Vh),
          frho(24 * (long)ctx->g.Vh)
    {
    }
    // the preconditioner's output in F32: SAP in F32 and the deflated SAP write it
    // directly, other forms are converted from their own output precision (the halves in use)
    lqcd_status precond_with(const lqcd_solver_params *p, const double2 *rho, T *ph)
    {
        const lqcd_sap_params &sap = p->sap;
        const int hs = nh == 1 ? 2 : 1;   // distance of the converted halves
        if (p->solver == LQCD_SOLVER_SAP_GCR && sap.prec != LQCD_F64) {
            void *a;
            const size_t fb = 2 * native_half_bytes(c, sap.prec) * nrhs;
            LQCD_TRY(ws_get(c, WS_SAP_IN, fb, &a));
            LQCD_TRY(convert_native(c, LQCD_F64, sap.prec, rho, a, 2 * nrhs));
            if (sap.prec == LQCD_F32) return sap_apply(c, &sap, a, ph, nrhs);
            void *b;
            LQCD_TRY(ws_get(c, WS_SAP_PSI, fb, &b));
            LQCD_TRY(sap_apply(c, &sap, a, b, nrhs));
            return convert_native(c, sap.prec, LQCD_F32, b, ph, nh * nrhs, hs, hs);
        }
        if (p->solver == LQCD_SOLVER_DFL_SAP_GCR) {
            bool done;
            LQCD_TRY(dfl_precond_native32(c, &sap, rho, ph, nh, nrhs, &done));
            if (done) return LQCD_OK;
        }
        void *t;
        LQCD_TRY(ws_get(c, WS_PHI64, (size_t)frho * nrhs * sizeof(double2), &t));
        LQCD_TRY(precond(c, p, rho, (double2 *)t, nrhs));
        return convert_native(c, LQCD_F64, LQCD_F32, t, ph, nh * nrhs, hs, hs);
    }
    lqcd_status D_inner(const T *ph, T *ch)
    {
        if (nh == 2) return dirac_D(c, LQCD_F32, ph, ch, nrhs);
        void *t;
        LQCD_TRY(ws_get(c, WS_TMP_O, native_half_bytes(c, LQCD_F32) * nrhs, &t));
        return dirac_dhat_s(c, LQCD_F32, ph, fphi, ch, fchi, t, nrhs);
    }
    lqcd_status dots(const T *A, const T *B, int kk, double *out)
    {
        return bdot32(c, fchi, nrhs, A, nrhs * fchi, fchi, B, fchi, kk, out);
    }
    lqcd_status axpy(int k, const double *cf, const T *X, T *y, double sign)
    {
        return bmulti_axpy32(c, fchi, nrhs, k, cf, X, nrhs * fchi, fchi, y, fchi, sign);
    }
    lqcd_status norm_rdot(const T *ch, const double2 *rho, double *out)
    {
        return bnorm_rdot32(c, nh, nrhs, ch, fchi, rho, frho, out);
    }
    lqcd_status rho_update(const double *cR, const double *s, T *ch, double2 *rho)
    {
        return brho_update32(c, nh, nrhs, cR, s, ch, fchi, rho, frho);
    }
    lqcd_status psi_update(int nk, const double *cf, const T *phi, double2 *psi)
    {
        return bmulti_axpy_mixed(c, nh, nrhs, nk, cf, phi, nrhs * fphi, fphi, psi, 12L * nh * c->g.Vh);
    }
    double final_fields() const { return 4.5; }
};

// flexible GCR on D psi_r = eta_r (nh = 2) or Dhat psi_r = eta_r (nh = 1) to
// |residual| <= tol |eta|; psi, eta: nrhs native FP64 fields of nh halves.
// warm: start from the given psi, which is zero otherwise.
template <class KV>
lqcd_status gcr_impl(lqcd_ctx *c, const lqcd_solver_params *sp, double tol, int nh, const double2 *eta,
                     double2 *psi, bool warm, int nrhs, int nmx, GcrState &S)
{
    using T = typename KV::T;
    KV kv(c, sp, nh, nrhs);
    const long Vh = c->g.Vh;
    const long ne = 12L * nh * Vh;   // double2 per FP64 field of nh halves
    const int nkv = sp->nkv;
    if (nkv < 1 || nkv > 64) return set_err(c, LQCD_ERR_ARG, "nkv=%d", nkv);
    if (nrhs * nkv > 1024 || nrhs > 64) return set_err(c, LQCD_ERR_ARG, "nrhs=%d with nkv=%d too large", nrhs, nkv);
    const long bphi = nrhs * kv.fphi, bchi = nrhs * kv.fchi;   // Krylov elements per batch of fields
    const size_t brho = (size_t)nrhs * kv.frho;
    void *buf;
    LQCD_TRY(ws_get(c, WS_SOLVER, nkv * (bphi + bchi) * sizeof(T) + (brho + nrhs * ne) * sizeof(double2), &buf));
    T *phi = (T *)buf, *chi = phi + nkv * bphi;
    double2 *rho = (double2 *)(chi + nkv * bchi), *w = rho + brho;
    const double inner_gain = sp->inner == LQCD_F64 ? 0.0 : 1e-5;
    const double gs_field = (double)bchi * sizeof(T);
    PhaseProf prof(c);
    std::vector<double> eta2(nrhs), rn2(nrhs), eta_n(nrhs), res(nrhs), cycle_start(nrhs);
    if (nh == 1) LQCD_TRY(blas_zero(c, brho * sizeof(double2), rho));
    // rho = eta - D psi (with_psi) or eta, and its norms
    auto residual = [&](bool with_psi, std::vector<double> &norms) -> lqcd_status {
        if (with_psi && nh == 2) LQCD_TRY(dirac_D(c, LQCD_F64, psi, w, nrhs));
        if (with_psi && nh == 1) {
            void *t;
            LQCD_TRY(ws_get(c, WS_TMP_O, native_half_bytes(c, LQCD_F64) * nrhs, &t));
            LQCD_TRY(dirac_dhat(c, LQCD_F64, psi, w, t, nrhs));
        }
        return bresidual64(c, nh, nrhs, eta, ne, with_psi ? w : nullptr, ne, rho, kv.frho, norms.data());
    };
    LQCD_TRY(residual(false, eta2));
    rn2 = eta2;
    if (warm) LQCD_TRY(residual(true, rn2));
    std::vector<char> active(nrhs);
    for (int r = 0; r < nrhs; r++) {
        eta_n[r] = std::sqrt(eta2[r]);
        res[r] = std::sqrt(rn2[r]);
        if (!std::isfinite(res[r])) S.status[r] = LQCD_ERR_NAN;
        else if (eta_n[r] == 0 || res[r] <= tol * eta_n[r]) S.status[r] = LQCD_OK;
        else S.status[r] = LQCD_ERR_NOT_CONVERGED;
        active[r] = S.status[r] == LQCD_ERR_NOT_CONVERGED;
    }
    // per rhs: a[r][i][k], b[r][k], cc[r][k], alpha[r][k]
    std::vector<Cplx> a((size_t)nrhs * nkv * nkv), cc((size_t)nrhs * nkv), alpha((size_t)nrhs * nkv);
    std::vector<double> b((size_t)nrhs * nkv), dots(2 * (size_t)nrhs * 64), coef(2 * (size_t)nrhs * 64);
    int it = 0;
    auto any_active = [&]() {
        for (int r = 0; r < nrhs; r++)
            if (active[r]) return true;
        return false;
    };
    while (any_active() && it < nmx) {
        int nk = 0;
        std::vector<char> done(nrhs, 0);
        for (int r = 0; r < nrhs; r++) cycle_start[r] = res[r];
        for (int k = 0; k < nkv && it < nmx; k++) {
            T *ph = phi + k * bphi, *ch = chi + k * bchi;
            prof.start();
            LQCD_TRY(kv.precond_with(sp, rho, ph));
            prof.stop(0);
            // chi_k = D phi_k, orthogonalised against chi_0..chi_{k-1}; leaves |chi_k|^2
            // and <rho, chi_k> in dots
            auto orth = [&]() -> lqcd_status {
                prof.start();
                LQCD_TRY(kv.D_inner(ph, ch));
                prof.stop(1);
                prof.start();
                for (int r = 0; r < nrhs; r++)
                    for (int i = 0; i < k; i++) a[((size_t)r * nkv + i) * nkv + k] = {0, 0};
                // classical Gram-Schmidt; a second pass only where the first removed more
                // than half of |chi_k|^2 (Daniel-Gragg-Kaufman-Stewart criterion).  The
                // first pass reduces chi_0..chi_k against chi_k, which also gives |chi_k|^2.
                for (int pass = 0; pass < 2 && k > 0; pass++) {
                    const int kk = pass == 0 ? k + 1 : k;
                    LQCD_TRY(kv.dots(chi, ch, kk, dots.data()));
                    bool again = false;
                    std::vector<double> cf(2 * (size_t)nrhs * k);
                    for (int r = 0; r < nrhs; r++) {
                        double removed = 0;
                        for (int i = 0; i < k; i++) {
                            const double dr = dots[2 * (r * kk + i)], di = dots[2 * (r * kk + i) + 1];
                            a[((size_t)r * nkv + i) * nkv + k].re += dr;
                            a[((size_t)r * nkv + i) * nkv + k].im += di;
                            cf[2 * (r * k + i)] = dr;
                            cf[2 * (r * k + i) + 1] = di;
                            removed += dr * dr + di * di;
                        }
                        if (pass == 0 && active[r] && removed > 0.5 * dots[2 * (r * kk + k)]) again = true;
                    }
                    LQCD_TRY(kv.axpy(k, cf.data(), chi, ch, -1.0));
                    // bytes: the dot reads kk + 1 fields, the update k + 1 and writes one
                    c->prof_gs_bytes += (kk + 1 + k + 2) * gs_field;
                    if (!again) break;
                    c->prof_gs_second += pass == 0;
                }
                return kv.norm_rdot(ch, rho, dots.data());
            };
            LQCD_TRY(orth());
            if (sp->solver == LQCD_SOLVER_NET_GCR || sp->solver == LQCD_SOLVER_DFL_NET_GCR) {
                // the network's direction must cut |rho| to 0.95 |rho| at least, i.e.
                // |c_k|^2 >= (1 - 0.95^2) |rho|^2; where it does not, SAP replaces it
                std::vector<int> reject;
                for (int r = 0; r < nrhs; r++) {
                    if (!active[r]) continue;
                    const double q2 = dots[2 * (2 * r)];
                    const double c2 = q2 > 0 ? (dots[2 * (2 * r + 1)] * dots[2 * (2 * r + 1)] +
                                                dots[2 * (2 * r + 1) + 1] * dots[2 * (2 * r + 1) + 1]) / q2
                                             : 0.0;
                    if (!std::isfinite(c2) || !std::isfinite(q2) || c2 < (1.0 - 0.95 * 0.95) * rn2[r]) reject.push_back(r);
                }
                if (!reject.empty()) {
                    void *fb;
                    LQCD_TRY(ws_get(c, WS_NET_FALLBACK, (size_t)bphi * sizeof(T), &fb));
                    lqcd_solver_params sap_only = *sp;
                    sap_only.solver = sp->solver == LQCD_SOLVER_DFL_NET_GCR ? LQCD_SOLVER_DFL_SAP_GCR
                                                                            : LQCD_SOLVER_SAP_GCR;
                    LQCD_TRY(kv.precond_with(&sap_only, rho, (T *)fb));
                    for (int r : reject) {
                        LQCD_CUDA_CHECK(c, cudaMemcpyAsync(ph + r * kv.fphi, (T *)fb + r * kv.fphi,
                                                           kv.fphi * sizeof(T), cudaMemcpyDeviceToDevice,
                                                           c->stream));
                        S.net_fallbacks[r]++;
                    }
                    LQCD_TRY(orth());
                }
            }
            std::vector<double> sx(nrhs);
            for (int r = 0; r < nrhs; r++) {
                const double bk = std::sqrt(dots[2 * (2 * r)]);
                b[(size_t)r * nkv + k] = bk;
                const double s = (bk > 0 && std::isfinite(bk)) ? 1.0 / bk : 0.0;
                if (active[r] && s == 0.0) {
                    S.status[r] = std::isfinite(bk) ? LQCD_ERR_BREAKDOWN : LQCD_ERR_NAN;
                    active[r] = 0;
                }
                // c_k = <chi_k / b_k, rho> = conj(<rho, chi_k>) / b_k
                const double cr = dots[2 * (2 * r + 1)] * s, ci = -dots[2 * (2 * r + 1) + 1] * s;
                cc[(size_t)r * nkv + k] = {cr, ci};
                // rho -= c_k chi_k / b_k (chi_k not yet normalised); chi_k *= 1/b_k
                coef[2 * r] = active[r] ? cr * s : 0.0;
                coef[2 * r + 1] = active[r] ? ci * s : 0.0;
                sx[r] = s;
                if (active[r]) rn2[r] = std::max(0.0, rn2[r] - (cr * cr + ci * ci));
            }
            LQCD_TRY(kv.rho_update(coef.data(), sx.data(), ch, rho));
            c->prof_gs_bytes += kv.final_fields() * (double)(nrhs * ne) * sizeof(double2);
            it++;
            nk = k + 1;
            bool recompute = false;
            for (int r = 0; r < nrhs; r++) {
                if (active[r]) S.iters[r]++;
                // |rho|^2 - |c|^2 loses digits once |rho| has dropped ~1e7 within the cycle
                if (active[r] && rn2[r] < 1e-14 * cycle_start[r] * cycle_start[r]) recompute = true;
            }
            if (recompute) {
                std::vector<double> d(2 * nrhs);
                LQCD_TRY(bblas_dot(c, 2 * ne, nrhs, (const double *)rho, 0, 2 * kv.frho, (const double *)rho,
                                   2 * kv.frho, 1, d.data()));
                for (int r = 0; r < nrhs; r++) rn2[r] = d[2 * r];
            }
            prof.stop(2);
            bool all_done = true;
            for (int r = 0; r < nrhs; r++) {
                double rr = std::sqrt(rn2[r]);
                if (!active[r] || rr <= tol * eta_n[r] || rr <= inner_gain * cycle_start[r]) done[r] = 1;
                all_done = all_done && done[r];
            }
            if (all_done) break;
        }
        // back substitution per rhs: alpha_j = (c_j - sum_{i>j} a_ji alpha_i) / b_j
        for (int r = 0; r < nrhs; r++) {
            for (int j = nk - 1; j >= 0; j--) {
                Cplx s = cc[(size_t)r * nkv + j];
                for (int i = j + 1; i < nk; i++) {
                    Cplx t = cmul(a[((size_t)r * nkv + j) * nkv + i], alpha[(size_t)r * nkv + i]);
                    s.re -= t.re;
                    s.im -= t.im;
                }
                double bj = b[(size_t)r * nkv + j];
                alpha[(size_t)r * nkv + j] = (active[r] && bj > 0) ? cdiv(s, bj) : Cplx{0, 0};
            }
            for (int j = 0; j < nk; j++) {
                coef[2 * (r * nk + j)] = alpha[(size_t)r * nkv + j].re;
                coef[2 * (r * nk + j) + 1] = alpha[(size_t)r * nkv + j].im;
            }
        }
        prof.start();
        if (nk > 0) LQCD_TRY(kv.psi_update(nk, coef.data(), phi, psi));
        // restart from the FP64 true residual
        LQCD_TRY(residual(true, rn2));
        prof.stop(3);
        for (int r = 0; r < nrhs; r++) {
            if (!active[r]) continue;
            res[r] = std::sqrt(rn2[r]);
            S.restarts[r]++;
            if (!std::isfinite(res[r])) {
                S.status[r] = LQCD_ERR_NAN;
                active[r] = 0;
            } else if (res[r] <= tol * eta_n[r]) {
                S.status[r] = LQCD_OK;
                active[r] = 0;
            }
        }
    }
    for (int r = 0; r < nrhs; r++) S.relres[r] = eta_n[r] > 0 ? res[r] / eta_n[r] : 0;
    return LQCD_OK;
}

// Krylov vectors in F64 or (krylov == F32, inner == F32) in F32
lqcd_status gcr_native(lqcd_ctx *c, const lqcd_solver_params *sp, int nh, const double2 *eta, double2 *psi, bool warm,
                       int nrhs, GcrState &S)
{
    if (sp->krylov == LQCD_F32) return gcr_impl<Krylov32>(c, sp, sp->tol, nh, eta, psi, warm, nrhs, sp->nmx, S);
    return gcr_impl<Krylov64>(c, sp, sp->tol, nh, eta, psi, warm, nrhs, sp->nmx, S);
}

lqcd_status check_params(lqcd_ctx *c, const lqcd_solver_params *p, int nrhs)
{
    if (!p || nrhs < 1) return set_err(c, LQCD_ERR_ARG, "bad solver arguments");
    if (!(p->tol > 0)) return set_err(c, LQCD_ERR_ARG, "tol must be > 0");
    if (!c->have_clover) return set_err(c, LQCD_ERR_STATE, "clover term not built");
    if ((p->solver == LQCD_SOLVER_DFL_SAP_GCR || p->solver == LQCD_SOLVER_DFL_NET_GCR) && !c->dfl)
        return set_err(c, LQCD_ERR_STATE, "deflation subspace not built");
    if ((p->solver == LQCD_SOLVER_NET_GCR || p->solver == LQCD_SOLVER_DFL_NET_GCR) && !c->net)
        return set_err(c, LQCD_ERR_STATE, "network not set");
    if (p->solver < LQCD_SOLVER_CGNR || p->solver > LQCD_SOLVER_DFL_NET_GCR)
        return set_err(c, LQCD_ERR_ARG, "solver %d", (int)p->solver);
    if (p->solver != LQCD_SOLVER_CGNR && (p->inner != LQCD_F64 && p->inner != LQCD_F32))
        return set_err(c, LQCD_ERR_ARG, "inner precision %d", (int)p->inner);
    if (p->krylov != LQCD_F64 && !(p->krylov == LQCD_F32 && p->inner == LQCD_F32))
        return set_err(c, LQCD_ERR_ARG, "Krylov precision %d with inner precision %d", (int)p->krylov,
                       (int)p->inner);
    return LQCD_OK;
}

lqcd_status worst(lqcd_status a, lqcd_status b) { return a != LQCD_OK ? a : b; }

// guess: psi holds the initial even-site guess x0 on entry (GCR solvers)
lqcd_status solve_dhat_impl(lqcd_ctx *c, const lqcd_solver_params *p, const double *eta, double *psi, int nrhs,
                            lqcd_solve_info *info, bool guess)
{
    if (!c || !eta || !psi) return set_err(c, LQCD_ERR_ARG, "null argument");
    LQCD_TRY(check_params(c, p, nrhs));
    if (guess && p->solver == LQCD_SOLVER_CGNR) return set_err(c, LQCD_ERR_ARG, "initial guesses are for the GCR solvers");
    const long Vh = c->g.Vh;
    const long nf = 24 * Vh;
    const size_t hb = native_half_bytes(c, LQCD_F64);
    lqcd_status all = LQCD_OK;
    double t0 = now_s();
    if (p->solver == LQCD_SOLVER_CGNR) {
        for (int k = 0; k < nrhs; k++) {
            lqcd_solve_info li{};
            void *io;
            LQCD_TRY(ws_get(c, WS_SOLVE_IO, 4 * hb, &io));
            double2 *eta_f = (double2 *)io, *psi_f = eta_f + nf;
            LQCD_TRY(blas_zero(c, 4 * hb, io));
            LQCD_TRY(pack_field(c, LQCD_F64, 1, eta + (size_t)k * 24 * Vh, eta_f, 1, false));
            lqcd_status st = cgnr_native(c, eta_f, psi_f, p->tol, p->nmx, &li);
            LQCD_TRY(pack_field(c, LQCD_F64, 1, psi + (size_t)k * 24 * Vh, psi_f, 1, true));
            if (info) info[k] = li;
            all = worst(all, st);
        }
    } else {
        // the even halves of every rhs, solved together
        void *io;
        LQCD_TRY(ws_get(c, WS_SOLVE_IO, 2 * hb * nrhs, &io));
        double2 *eta_e = (double2 *)io, *psi_e = eta_e + nrhs * 12 * Vh;
        LQCD_TRY(pack_field(c, LQCD_F64, 1, eta, eta_e, nrhs, false));
        if (guess)
            LQCD_TRY(pack_field(c, LQCD_F64, 1, psi, psi_e, nrhs, false));
        else
            LQCD_TRY(blas_zero(c, hb * nrhs, psi_e));
        GcrState S(nrhs);
        LQCD_TRY(gcr_native(c, p, 1, eta_e, psi_e, guess, nrhs, S));
        LQCD_TRY(pack_field(c, LQCD_F64, 1, psi, psi_e, nrhs, true));
        for (int k = 0; k < nrhs; k++) {
            if (info) {
                info[k].iters = S.iters[k];
                info[k].restarts = S.restarts[k];
                // with psi_o = -A_oo^-1 H_oe psi_e the residual of D is that of Dhat
                info[k].true_relres = S.relres[k];
                info[k].relres_dhat = S.relres[k];
                info[k].status = S.status[k];
                info[k].seconds = now_s() - t0;
                info[k].net_fallbacks = S.net_fallbacks[k];
            }
            all = worst(all, S.status[k]);
        }
    }
    if (all != LQCD_OK && all != LQCD_ERR_CUDA) set_err(c, all, "solve did not converge (status %d)", (int)all);
    return all;
}

}  // namespace

extern "C" {

lqcd_status lqcd_solve_dhat(lqcd_ctx *c, const lqcd_solver_params *p, const double *eta, double *psi, int nrhs,
                            lqcd_solve_info *info)
{
    return solve_dhat_impl(c, p, eta, psi, nrhs, info, false);
}

lqcd_status lqcd_solve_dhat_guess(lqcd_ctx *c, const lqcd_solver_params *p, const double *eta, double *psi,
                                  int nrhs, lqcd_solve_info *info)
{
    return solve_dhat_impl(c, p, eta, psi, nrhs, info, true);
}

lqcd_status lqcd_solve_D(lqcd_ctx *c, const lqcd_solver_params *p, const double *eta, double *psi, int nrhs,
                         lqcd_solve_info *info)
{
    if (!c || !eta || !psi) return set_err(c, LQCD_ERR_ARG, "null argument");
    LQCD_TRY(check_params(c, p, nrhs));
    if (p->solver == LQCD_SOLVER_CGNR) return set_err(c, LQCD_ERR_ARG, "CGNR solves Dhat only");
    const long Vh = c->g.Vh;
    const long nf = 24 * Vh;
    const size_t hb = native_half_bytes(c, LQCD_F64);
    double t0 = now_s();
    void *io;
    LQCD_TRY(ws_get(c, WS_SOLVE_IO, 4 * hb * nrhs, &io));
    double2 *eta_f = (double2 *)io, *psi_f = eta_f + nrhs * nf;
    LQCD_TRY(pack_field(c, LQCD_F64, 2, eta, eta_f, nrhs, false));
    LQCD_TRY(blas_zero(c, 2 * hb * nrhs, psi_f));
    GcrState S(nrhs);
    LQCD_TRY(gcr_native(c, p, 2, eta_f, psi_f, false, nrhs, S));
    LQCD_TRY(pack_field(c, LQCD_F64, 2, psi, psi_f, nrhs, true));
    lqcd_status all = LQCD_OK;
    for (int k = 0; k < nrhs; k++) {
        if (info) {
            info[k].iters = S.iters[k];
            info[k].restarts = S.restarts[k];
            info[k].true_relres = S.relres[k];
            info[k].relres_dhat = -1;
            info[k].status = S.status[k];
            info[k].seconds = now_s() - t0;
            info[k].net_fallbacks = S.net_fallbacks[k];
        }
        all = worst(all, S.status[k]);
    }
    return all;
}

}  // extern "C"
