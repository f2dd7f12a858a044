// Even-odd CG on the normal equation, Dhat^dag Dhat psi = Dhat^dag eta (Eq. 2),
// FP64, with its scalars on the device.
//
// On small lattices an iteration is a handful of kernels of a few microseconds;
// what it spent most on was the host: three waits per iteration for a norm and
// the launches behind each.  Here every kernel that needs a scalar sums the
// partial norms of the kernel before it (a fixed order, the same in every CTA),
// the stopping test runs on the device, and the host stays ahead: an iteration
// past the end finds the state closed and changes nothing.  gamma5 is applied in
// the updates, so that Dhat^dag = gamma5 Dhat gamma5 costs no pass of its own.
//
// An iteration past the end still costs its two Dhat, so the host sends one unit
// (an iteration, or a graph) beyond the one it waits for, and only while the mean
// decay of the residual so far puts the end behind it: solves of one to four
// iterations took up to twice the time with two units always ahead (16384 even
// sites, one iteration: 1820 us; 549 us now; 861 us with the scalars on the host).
// On lattices of up to CG_GRAPH_SITES even sites, where launching takes as long as
// the kernels, four iterations are captured as a graph once CG_GRAPH_FROM are
// expected, on a stream of the context's own (a legacy default stream cannot be
// captured).  Making the graph takes about 250 us; an iteration costs, with plain
// launches / in graphs, at 2048 even sites 61 / 50 us, 4096 98 / 74, 8192 173 / 120,
// 16384 220 / 205.  131 iterations on 8^4: 16.0 -> 6.7 ms (with the state copied to the
// host instead of written there 8.7 ms).
#include <cmath>

#include "lqcd_internal.cuh"

namespace {

constexpr int CG_THREADS = 256;
constexpr int CG_RING = 4;      // states in flight; iterations of a graph
constexpr int CG_GRAPH_SITES = 16384;   // even sites
constexpr int CG_GRAPH_FROM = 16;       // iterations still to come

enum { CG_RUN = 0, CG_BELOW, CG_BREAKDOWN, CG_NAN };

struct CgState {
    double zz;      // |z|^2 of the current direction
    double rr;      // |r|^2 (recursive)
    int code;       // CG_RUN, or why the iteration ended
    int iters;
};

// sum of nb partials in a fixed order, in every thread of the CTA
__device__ __forceinline__ double part_sum(const double *part, int nb)
{
    __shared__ double sh[CG_THREADS / 32];
    double v[1] = {0};
    for (int i = threadIdx.x; i < nb; i += CG_THREADS) v[0] += part[i];
    warp_multi_sum(v);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v[0];
    __syncthreads();
    double s = 0;
    for (int w = 0; w < CG_THREADS / 32; w++) s += sh[w];
    return s;
}
__device__ __forceinline__ void part_store(double x, double *part)
{
    __shared__ double sh[CG_THREADS / 32];
    double v[1] = {x};
    warp_multi_sum(v);
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v[0];
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int w = 0; w < CG_THREADS / 32; w++) s += sh[w];
        part[blockIdx.x] = s;
    }
}
// sign flip of the lower spins (entries from 6 Vh on), off the FP64 pipe
__device__ __forceinline__ double2 g5(double2 v, bool low)
{
    const int m = low ? (int)0x80000000u : 0;
    return make_double2(__hiloint2double(__double2hiint(v.x) ^ m, __double2loint(v.x)),
                        __hiloint2double(__double2hiint(v.y) ^ m, __double2loint(v.y)));
}

__global__ void __launch_bounds__(CG_THREADS) k_cg_norm(long n, const double2 *__restrict__ w, double *part)
{
    after_previous();
    double s = 0;
#pragma unroll 4
    for (long j = blockIdx.x * (long)CG_THREADS + threadIdx.x; j < n; j += (long)gridDim.x * CG_THREADS)
        s = norm_add(s, w[j]);
    part_store(s, part);
}

// alpha = zz / |w|^2; x += alpha p, r -= alpha w, t = gamma5 r, partial |r|^2
__global__ void __launch_bounds__(CG_THREADS) k_cg_xr(long n, int nb, const CgState *S, const double *pw,
                                                      const double2 *__restrict__ p, const double2 *__restrict__ w,
                                                      double2 *x, double2 *r, double2 *t, double *prr)
{
    after_previous();
    if (S->code != CG_RUN) return;
    const double ww = part_sum(pw, nb);
    if (!(ww > 0) || !isfinite(ww)) return;   // k_cg_p closes the state
    const double al = S->zz / ww;
    double s = 0;
#pragma unroll 2
    for (long j = blockIdx.x * (long)CG_THREADS + threadIdx.x; j < n; j += (long)gridDim.x * CG_THREADS) {
        const double2 pj = p[j], wj = w[j], xj = x[j], rj = r[j];
        x[j] = make_double2(fmx(al, pj.x, xj.x), fmx(al, pj.y, xj.y));
        const double2 q = make_double2(fmx(-al, wj.x, rj.x), fmx(-al, wj.y, rj.y));
        r[j] = q;
        t[j] = g5(q, 2 * j >= n);
        s = norm_add(s, q);
    }
    part_store(s, prr);
}

// z = gamma5 zp; beta = |z|^2 / zz; p = z + beta p; the state of the next iteration
// goes to Sn (S is read by every CTA of this launch) and to Hn in pinned host
// memory (a copy of its own would cost more than this kernel)
__global__ void __launch_bounds__(CG_THREADS) k_cg_p(long n, int nb, const CgState *S, CgState *Sn, CgState *Hn,
                                                     double tol2,
                                                     const double *pw, const double *prr, const double *pzz,
                                                     const double2 *__restrict__ zp, double2 *p)
{
    after_previous();
    CgState s = *S;
    if (s.code == CG_RUN) {
        const double ww = part_sum(pw, nb);
        if (!isfinite(ww)) {
            s.code = CG_NAN;
        } else if (!(ww > 0)) {
            s.code = CG_BREAKDOWN;
        } else {
            s.rr = part_sum(prr, nb);
            s.iters++;
            if (s.rr <= tol2) s.code = CG_BELOW;
        }
        if (s.code == CG_RUN) {
            const double zz = part_sum(pzz, nb), beta = zz / s.zz;
#pragma unroll 2
            for (long j = blockIdx.x * (long)CG_THREADS + threadIdx.x; j < n; j += (long)gridDim.x * CG_THREADS) {
                const double2 z = g5(zp[j], 2 * j >= n), q = p[j];
                p[j] = make_double2(fmx(beta, q.x, z.x), fmx(beta, q.y, z.y));
            }
            s.zz = zz;
        }
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *Sn = s;
        *Hn = s;
    }
}

}  // namespace

namespace {

struct CgEvents {
    cudaEvent_t e[2] = {};
    ~CgEvents()
    {
        for (cudaEvent_t v : e)
            if (v) cudaEventDestroy(v);
    }
};
// the solve on the context's own stream, ordered after and before the caller's
struct CgStream {
    lqcd_ctx *c;
    cudaStream_t user;
    cudaEvent_t ev = nullptr;
    cudaGraphExec_t graph = nullptr;
    bool on = false, failed = false;
    explicit CgStream(lqcd_ctx *ctx) : c(ctx), user(ctx->stream) {}
    lqcd_status enter()
    {
        if (!c->cg_stream) LQCD_CUDA_CHECK(c, cudaStreamCreateWithFlags(&c->cg_stream, cudaStreamNonBlocking));
        LQCD_CUDA_CHECK(c, cudaEventCreateWithFlags(&ev, cudaEventDisableTiming));
        LQCD_CUDA_CHECK(c, cudaEventRecord(ev, user));
        LQCD_CUDA_CHECK(c, cudaStreamWaitEvent(c->cg_stream, ev, 0));
        c->stream = c->cg_stream;
        on = true;
        return LQCD_OK;
    }
    ~CgStream()
    {
        if (on) {
            cudaEventRecord(ev, c->stream);
            cudaStreamWaitEvent(user, ev, 0);
            c->stream = user;
        }
        if (graph) cudaGraphExecDestroy(graph);
        if (ev) cudaEventDestroy(ev);
    }
};

}  // namespace

// eta, x: native FP64 even fields; x is set to the solution
lqcd_status cgnr_native(lqcd_ctx *c, const double2 *eta, double2 *x, double tol, int nmx, lqcd_solve_info *info)
{
    const long Vh = c->g.Vh, n = 12 * Vh, n2 = 2 * n;
    const size_t hb = native_half_bytes(c, LQCD_F64);
    const int nb = (int)std::max<long>(1, std::min<long>(4 * 152, (n + CG_THREADS - 1) / CG_THREADS));
    const double t0 = ProfClock::wall();
    void *buf, *tmp_o;
    LQCD_TRY(ws_get(c, WS_CGNR, 5 * hb + 3 * nb * sizeof(double) + CG_RING * sizeof(CgState), &buf));
    double2 *r = (double2 *)buf, *z = r + n, *p = z + n, *w = p + n, *t = w + n;
    double *pw = (double *)(t + n), *prr = pw + nb, *pzz = prr + nb;
    CgState *S = (CgState *)(pzz + nb);      // a ring: iteration i reads i and writes i + 1
    CgState *H = (CgState *)c->red_host;     // pinned: what iteration i wrote at i, the start at CG_RING
    LQCD_TRY(ws_get(c, WS_TMP_O, hb, &tmp_o));
    auto dhat = [&](const double2 *in, double2 *out) { return dirac_dhat(c, LQCD_F64, in, out, tmp_o, 1); };
    auto dhat_dag = [&](const double2 *in, double2 *out) -> lqcd_status {
        LQCD_TRY(blas_gamma5_native64(c, 1, in, t));
        LQCD_TRY(dhat(t, out));
        return blas_gamma5_native64(c, 1, out, out);
    };
    CgEvents ev;
    for (cudaEvent_t &v : ev.e) LQCD_CUDA_CHECK(c, cudaEventCreateWithFlags(&v, cudaEventDisableTiming));
    CgStream own(c);
    if (Vh <= CG_GRAPH_SITES) LQCD_TRY(own.enter());
    LQCD_TRY(blas_zero(c, hb, x));
    LQCD_TRY(blas_copy(c, n2, (const double *)eta, (double *)r));
    double eta2;
    LQCD_TRY(blas_norm2(c, n2, (const double *)eta, &eta2));
    const double tol2 = tol * tol * eta2;
    // iteration i of a start: p -> x, r, p, state i -> i + 1
    auto iteration = [&](long i) -> lqcd_status {
        CgState *cur = S + i % CG_RING, *nxt = S + (i + 1) % CG_RING;
        const bool pdl = !c->capturing;
        LQCD_TRY(dhat(p, w));
        launch_pdl(pdl, k_cg_norm, nb, CG_THREADS, c->stream, n, w, pw);
        launch_pdl(pdl, k_cg_xr, nb, CG_THREADS, c->stream, n, nb, cur, pw, p, w, x, r, t, prr);
        LQCD_TRY(dhat(t, z));
        launch_pdl(pdl, k_cg_norm, nb, CG_THREADS, c->stream, n, z, pzz);
        launch_pdl(pdl, k_cg_p, nb, CG_THREADS, c->stream, n, nb, cur, nxt, H + i % CG_RING, tol2, pw, prr, pzz, z, p);
        c->n_kernel_launches += 4;
        LQCD_LAUNCH_CHECK(c);
        return LQCD_OK;
    };
    // CG_RING iterations as a graph; without it plain launches serve
    auto make_graph = [&]() -> lqcd_status {
        cudaGraph_t g = nullptr;
        const long before = c->n_kernel_launches;
        c->capturing = true;
        lqcd_status cs = LQCD_OK;
        bool ok = cudaStreamBeginCapture(c->stream, cudaStreamCaptureModeThreadLocal) == cudaSuccess;
        if (ok) {
            for (int i = 0; i < CG_RING && cs == LQCD_OK; i++) cs = iteration(i);
            ok = cudaStreamEndCapture(c->stream, &g) == cudaSuccess && cs == LQCD_OK && g &&
                 cudaGraphInstantiate(&own.graph, g, 0) == cudaSuccess;
        }
        c->capturing = false;
        c->n_kernel_launches = before;   // recorded, not run
        if (g) cudaGraphDestroy(g);
        if (!ok) {
            cudaGetLastError();
            own.graph = nullptr;
            own.failed = true;
        }
        return LQCD_OK;
    };
    int it = 0;
    lqcd_status st = LQCD_ERR_NOT_CONVERGED;
    double rr = eta2;
    if (eta2 == 0) {
        st = LQCD_OK;
    } else if (!std::isfinite(eta2)) {
        st = LQCD_ERR_NAN;
    } else {
        while (st == LQCD_ERR_NOT_CONVERGED && it < nmx) {
            // (re)start from the residual in r
            CgState s0{};
            LQCD_TRY(dhat_dag(r, z));
            LQCD_TRY(blas_copy(c, n2, (const double *)z, (double *)p));
            LQCD_TRY(blas_norm2(c, n2, (const double *)z, &s0.zz));
            s0.iters = it;
            H[CG_RING] = s0;
            LQCD_CUDA_CHECK(c, cudaMemcpyAsync(S, H + CG_RING, sizeof(CgState), cudaMemcpyHostToDevice, c->stream));
            const long limit = (long)nmx - it;
            const double rr0 = rr;
            CgState last = s0;
            last.rr = rr0;
            long sent = 0, seen = 0;   // iterations of this start launched / whose state is known
            long end[2] = {0, 0};      // of the units in flight: a graph, or one iteration
            int first = 0, flying = 0;
            // Iterations still to come by the mean decay so far (CGNR's residual never
            // grows; its decay slows down, so the estimate is rather too small).
            auto left = [&]() -> double {
                const int k = last.iters - s0.iters;
                const double d = k > 0 ? std::log(rr0 / last.rr) : 0;
                return d > 0 ? k * std::log(last.rr / tol2) / d : 0;
            };
            auto send = [&]() -> lqcd_status {
                const double more = std::min(left(), (double)(limit - seen)) - (sent - seen);
                if (own.on && !own.graph && !own.failed && more >= CG_GRAPH_FROM) LQCD_TRY(make_graph());
                if (own.graph && sent % CG_RING == 0 && more >= CG_RING) {
                    LQCD_CUDA_CHECK(c, cudaGraphLaunch(own.graph, c->stream));
                    c->n_kernel_launches += 8 * CG_RING;
                    sent += CG_RING;
                } else {
                    LQCD_TRY(iteration(sent));
                    sent++;
                }
                const int u = (first + flying++) % 2;
                end[u] = sent;
                LQCD_CUDA_CHECK(c, cudaEventRecord(ev.e[u], c->stream));
                return LQCD_OK;
            };
            while (last.code == CG_RUN && seen < limit) {
                if (flying == 0) LQCD_TRY(send());
                // a second unit while the end is expected behind the first
                if (flying == 1 && sent < limit && left() >= (double)(sent - seen + 1)) LQCD_TRY(send());
                LQCD_CUDA_CHECK(c, cudaEventSynchronize(ev.e[first]));
                seen = end[first];
                first = (first + 1) % 2;
                flying--;
                // a graph in flight may have overwritten it: with a later state of this
                // start, and a closed one stays as it is
                volatile CgState *h = H + (seen - 1) % CG_RING;
                last.code = h->code;
                last.rr = h->rr;
                last.iters = h->iters;
            }
            LQCD_CUDA_CHECK(c, cudaStreamSynchronize(c->stream));   // iterations past the end are no-ops
            last = H[(sent - 1) % CG_RING];
            const bool moved = last.iters > it;
            it = last.iters;
            rr = last.rr;
            if (last.code == CG_NAN) st = LQCD_ERR_NAN;
            if (last.code == CG_BREAKDOWN) st = LQCD_ERR_BREAKDOWN;
            if (last.code != CG_BELOW || !moved) break;   // no start without an iteration is repeated
            // recompute the residual before accepting; too large: another start from it
            LQCD_TRY(dhat(x, w));
            LQCD_TRY(blas_sub(c, n2, (const double *)eta, (const double *)w, (double *)r));
            LQCD_TRY(blas_norm2(c, n2, (const double *)r, &rr));
            if (rr <= tol2) st = LQCD_OK;
        }
    }
    // final true residual
    if (st != LQCD_OK || eta2 == 0) {
        LQCD_TRY(dhat(x, w));
        LQCD_TRY(blas_sub(c, n2, (const double *)eta, (const double *)w, (double *)r));
        LQCD_TRY(blas_norm2(c, n2, (const double *)r, &rr));
    }
    if (info) {
        info->iters = it;
        info->restarts = 0;
        info->relres_dhat = eta2 > 0 ? std::sqrt(rr / eta2) : 0;
        info->true_relres = info->relres_dhat;
        info->seconds = ProfClock::wall() - t0;
        info->status = st;
    }
    return st;
}
