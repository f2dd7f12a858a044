// Internal declarations of the sm_103a Wilson-clover library: context,
// device-private ("native") layouts, geometry and the chiral-basis spin
// algebra of the hopping term (Eq. 1).
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cstdint>
#include <cstdio>
#include <ctime>
#include <string>
#include <vector>

#include "lqcd.h"

// ------------------------------------------------------------------ complex
template <class R>
struct cx {
    R re, im;
};
template <class R>
__host__ __device__ __forceinline__ cx<R> mk(R a, R b) { return cx<R>{a, b}; }
template <class R>
__device__ __forceinline__ cx<R> operator+(cx<R> a, cx<R> b) { return {a.re + b.re, a.im + b.im}; }
template <class R>
__device__ __forceinline__ cx<R> operator-(cx<R> a, cx<R> b) { return {a.re - b.re, a.im - b.im}; }
template <class R>
__device__ __forceinline__ cx<R> operator-(cx<R> a) { return {-a.re, -a.im}; }
template <class R>
__device__ __forceinline__ cx<R> operator*(cx<R> a, cx<R> b)
{
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <class R>
__device__ __forceinline__ cx<R> operator*(R s, cx<R> a) { return {s * a.re, s * a.im}; }
template <class R>
__device__ __forceinline__ cx<R> conjx(cx<R> a) { return {a.re, -a.im}; }
template <class R>
__device__ __forceinline__ cx<R> timesI(cx<R> a) { return {-a.im, a.re}; }   // i a
template <class R>
__device__ __forceinline__ cx<R> timesmI(cx<R> a) { return {a.im, -a.re}; }  // -i a
// a * b with a conjugated
template <class R>
__device__ __forceinline__ cx<R> cmulc(cx<R> a, cx<R> b)
{
    return {a.re * b.re + a.im * b.im, a.re * b.im - a.im * b.re};
}

// a * b + c with a single rounding
__device__ __forceinline__ float fmx(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fmx(double a, double b, double c) { return __fma_rn(a, b, c); }

// (re, im) += conj(a) b and += c x with one fused multiply-add per real product
// (a sum of products written out compiles to a product, a fused multiply-add
// and an addition: half as much again on the FP64 pipe that bounds FP64 BLAS)
__device__ __forceinline__ void cdot_add(double &re, double &im, double2 a, double2 b)
{
    re = fmx(a.x, b.x, re);
    re = fmx(a.y, b.y, re);
    im = fmx(a.x, b.y, im);
    im = fmx(-a.y, b.x, im);
}
__device__ __forceinline__ double2 caxpy(double2 c, double2 x, double2 y)   // y + c x
{
    y.x = fmx(c.x, x.x, y.x);
    y.x = fmx(-c.y, x.y, y.x);
    y.y = fmx(c.x, x.y, y.y);
    y.y = fmx(c.y, x.x, y.y);
    return y;
}
__device__ __forceinline__ double norm_add(double n, double2 a) { return fmx(a.y, a.y, fmx(a.x, a.x, n)); }

// Warp sums of V = 1, 2, 4, 8 or 16 values in V - 1 + 5 - log2 V additions (a
// butterfly over each takes 5 V): in each step a lane hands half of its values
// to its partner and adds the partner's other half to what it keeps.  On
// return v[0] is the sum of value lane * V / 32.
template <int V>
__device__ __forceinline__ void warp_multi_sum(double (&v)[V])
{
    const int lane = threadIdx.x & 31;
    int off = 16;
#pragma unroll
    for (int h = V / 2; h >= 1; h /= 2, off /= 2) {
        const bool up = lane & off;
#pragma unroll
        for (int j = 0; j < h; j++) {
            const double send = up ? v[j] : v[j + h];
            v[j] = (up ? v[j + h] : v[j]) + __shfl_xor_sync(0xffffffffu, send, off);
        }
    }
#pragma unroll
    for (; off > 0; off /= 2) v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
}

// double <-> float of N numbers in integer arithmetic, the same values as the casts.
// A cast takes a slot of the FP64 pipe (2 a clock and SM), eight integer
// instructions a sixteenth of the chip's rate: with 24 casts per site each way a
// conversion pass is bound by the pipe and not by memory.  Numbers outside float's
// normal range (zero, too) send all N through the casts.
template <int N>
__device__ __forceinline__ void narrow(const double (&x)[N], float (&f)[N])
{
    bool odd = false;
#pragma unroll
    for (int i = 0; i < N; i++) {
        const unsigned hi = __double2hiint(x[i]), lo = __double2loint(x[i]), t = hi & 0x7fffffffu;
        odd |= t - 0x38100000u >= 0x0fe00000u;   // |x| < 2^-126 or >= 2^128
        // mantissa cut to 23 bits, then rounded to nearest, ties to even (a carry
        // runs on into the exponent)
        unsigned u = __funnelshift_l(lo, t - 0x38000000u, 3);
        u += ((lo & 0x1fffffffu) + (u & 1u) + 0x0fffffffu) >> 29;
        f[i] = __uint_as_float(u | (hi & 0x80000000u));
    }
    if (odd) {
        asm volatile("");   // a branch: the compiler would rather run the casts always
#pragma unroll
        for (int i = 0; i < N; i++) f[i] = (float)x[i];
    }
}
template <int N>
__device__ __forceinline__ void widen(const float (&f)[N], double (&x)[N])
{
    bool odd = false;
#pragma unroll
    for (int i = 0; i < N; i++) {
        const unsigned u = __float_as_uint(f[i]), t = u & 0x7fffffffu;
        odd |= t - 0x00800000u >= 0x7f000000u;   // zero, subnormal, infinite, NaN
        x[i] = __hiloint2double((int)((u & 0x80000000u) | ((t >> 3) + 0x38000000u)), (int)(u << 29));
    }
    if (odd) {
        asm volatile("");
#pragma unroll
        for (int i = 0; i < N; i++) x[i] = f[i];
    }
}

// third row of an SU(3) matrix from the first two, u2 = (u0 x u1)^*, each real
// part one product and three fused multiply-adds
template <class R>
__device__ __forceinline__ void su3_third_row(cx<R> u[3][3])
{
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const int k = (j + 1) % 3, l = (j + 2) % 3;
        const cx<R> a = u[0][k], b = u[1][l], c = u[0][l], d = u[1][k];
        // conj(a b - c d)
        R re = a.re * b.re;
        re = fmx(-a.im, b.im, re);
        re = fmx(-c.re, d.re, re);
        re = fmx(c.im, d.im, re);
        R im = -a.re * b.im;
        im = fmx(-a.im, b.re, im);
        im = fmx(c.re, d.im, im);
        im = fmx(c.im, d.re, im);
        u[2][j] = mk(re, im);
    }
}

// ------------------------------------------------------------------ geometry
// Division of a non-negative 31-bit n by an invariant d >= 1 as a multiply-high,
// an add and a shift (Granlund & Montgomery, "Division by invariant integers
// using multiplication", 1994, round-up method): with l = ceil(log2 d) and
// m = floor(2^32 (2^l - d) / d) + 1, n / d = (mulhi(m, n) + n) >> l exactly for
// 0 <= n < 2^31 (mulhi(m, n) < n, so the sum does not overflow 32 bits).
struct FastDiv {
    unsigned m;
    int l;
};
inline FastDiv make_fastdiv(int d)
{
    int l = 0;
    while ((1u << l) < (unsigned)d) l++;
    const unsigned long long m =
        ((1ull << 32) * ((1ull << l) - (unsigned long long)d)) / (unsigned long long)d + 1;
    return FastDiv{(unsigned)m, l};
}
__device__ __forceinline__ int fast_div(const FastDiv &f, int n)
{
    return (int)((__umulhi(f.m, (unsigned)n) + (unsigned)n) >> f.l);
}

struct Geom {
    int L[4];      // L[0] = T
    int V, Vh;
    int L3h;       // L3 / 2
    int bc_t;      // -1 antiperiodic fermion field in time, +1 periodic
    FastDiv dL3h, dL2, dL1;   // divisions by L3h, L[2], L[1]
};
// fills the derived fields of a geometry from its extents
void geom_init(Geom &g, const int L[4], int bc_t);

// coordinates of the site of parity p and rank r (site = 2r + b)
__device__ __forceinline__ void rank_coords(const Geom &g, int p, int r, int x[4])
{
    const int row = fast_div(g.dL3h, r);
    const int x3h = r - row * g.L3h;
    const int t = fast_div(g.dL2, row);
    x[2] = row - t * g.L[2];
    x[0] = fast_div(g.dL1, t);
    x[1] = t - x[0] * g.L[1];
    const int b = (p + x[0] + x[1] + x[2]) & 1;
    x[3] = 2 * x3h + b;
}
__device__ __forceinline__ int coords_rank(const Geom &g, const int x[4])
{
    return (x[3] + g.L[3] * (x[2] + g.L[2] * (x[1] + g.L[1] * x[0]))) >> 1;
}
// rank of the neighbour x + d*mu (d = +-1), periodic wrap
__device__ __forceinline__ int nbr_rank(const Geom &g, const int x[4], int mu, int d)
{
    int y[4] = {x[0], x[1], x[2], x[3]};
    int v = y[mu] + d;
    y[mu] = v < 0 ? v + g.L[mu] : (v >= g.L[mu] ? v - g.L[mu] : v);
    return coords_rank(g, y);
}

// ------------------------------------------------------------------ context
struct Workspace {
    void *p = nullptr;
    size_t bytes = 0;
};

// the autotuner's choice for a stencil launch, kept with the context while nothing
// it depends on changes (building and looking up its key took longer than the
// launch)
constexpr int TUNE_SLOTS = 4;   // calls with one and with several right-hand sides take turns
struct TuneMemo {
    long gen = -1;      // generation of the tuner's table
    int nrhs = 0, force = 0;
    int variant = 0, tx = 0, ty = 0, nr = 0, kind = 0;
};

// the same for an operator: are its kernels launched dependently?
struct DepMemo {
    long gen = -1;
    int nrhs = 0;
    bool dep = true;
};

struct DflState;   // deflation subspace (lqcd_dfl.cu)
struct NetState;   // learned preconditioner (lqcd_ptc.cu)
struct ChronoState;   // stored solutions for initial guesses (lqcd_chrono.cu)

struct lqcd_ctx {
    lqcd_geom geom;
    Geom g;
    cudaStream_t stream = nullptr;
    char err[512] = {0};
    // gauge field, native layouts
    double2 *U64 = nullptr;   // [p][mu][9][Vh]      full SU(3), FP64
    float4 *U32 = nullptr;    // [p][mu][3][Vh]      two rows, FP32
    uint2 *U16 = nullptr;     // [p][mu][3][Vh]      two rows, FP16 (4 halves per uint2)
    bool have_gauge = false;
    // clover term: A and A^-1 for both parities, packed Hermitian 6x6 pairs
    double2 *A64[2] = {nullptr, nullptr}, *Ai64[2] = {nullptr, nullptr};  // [36][Vh]
    float4 *A32[2] = {nullptr, nullptr}, *Ai32[2] = {nullptr, nullptr};   // [18][Vh]
    uint2 *A16[2] = {nullptr, nullptr}, *Ai16[2] = {nullptr, nullptr};    // [18][Vh], FP16
    bool have_clover = false;
    long op_version = 0;   // changes with the links and with the clover term
    double kappa = 0, csw = 0;
    double logdet_e = 0, logdet_o = 0;   // log|det A| of each parity, from the last clover build
    // device scratch for reductions
    double *red = nullptr;        // partial sums
    double *red_out = nullptr;    // final reduction results (device)
    double *red_host = nullptr;   // pinned host mirror
    // named temporary buffers, grown on demand
    Workspace ws[24];   // indexed by the WS_ slots below
    DflState *dfl = nullptr;
    NetState *net = nullptr;
    ChronoState *chrono = nullptr;
    long n_kernel_launches = 0;
    TuneMemo tune[4][3][2][TUNE_SLOTS];   // [mode][precision][output parity][nrhs % TUNE_SLOTS]
    DepMemo dep[2][3][TUNE_SLOTS];        // [Dhat, D][precision][nrhs % TUNE_SLOTS]
    bool hop_dep = true;      // the choice for the stencil launches of the operator under way
    bool capturing = false;               // launches go into a graph being captured
    cudaStream_t cg_stream = nullptr;     // CGNR on small lattices (lqcd_cgnr.cu)
    // LQCD_PROFILE=1: synchronised wall time of solver phases, reported on
    // stderr by the GCR (developer instrumentation; off by default)
    bool prof_on = false;
    double prof_t[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    double prof_gs_bytes = 0;   // algorithmic bytes of the outer Gram-Schmidt
    long prof_gs_second = 0;    // second Gram-Schmidt passes taken
};

// laps of the LQCD_PROFILE clock: lap(i) adds the time since the previous lap
// (or construction) to c->prof_t[i]; nothing happens when profiling is off
struct ProfClock {
    lqcd_ctx *c;
    double t0 = 0;
    static double wall()
    {
        timespec ts;
        clock_gettime(CLOCK_MONOTONIC, &ts);
        return ts.tv_sec + 1e-9 * ts.tv_nsec;
    }
    explicit ProfClock(lqcd_ctx *ctx) : c(ctx)
    {
        if (!c->prof_on) return;
        cudaStreamSynchronize(c->stream);
        t0 = wall();
    }
    void lap(int i)
    {
        if (!c->prof_on) return;
        cudaStreamSynchronize(c->stream);
        const double t = wall();
        c->prof_t[i] += t - t0;
        t0 = t;
    }
};

// error helpers
lqcd_status set_err(lqcd_ctx *c, lqcd_status s, const char *fmt, ...);
#define LQCD_CUDA_CHECK(ctx, call)                                                          \
    do {                                                                                    \
        cudaError_t e__ = (call);                                                           \
        if (e__ != cudaSuccess)                                                             \
            return set_err(ctx, LQCD_ERR_CUDA, "%s:%d %s: %s", __FILE__, __LINE__, #call,   \
                           cudaGetErrorString(e__));                                        \
    } while (0)
#define LQCD_LAUNCH_CHECK(ctx) LQCD_CUDA_CHECK(ctx, cudaGetLastError())
#define LQCD_TRY(expr)                         \
    do {                                       \
        lqcd_status s__ = (expr);              \
        if (s__ != LQCD_OK) return s__;        \
    } while (0)

// workspace slots
enum {
    WS_PACK_IN = 0,
    WS_PACK_OUT,
    WS_TMP_O,       // odd temporaries of Dhat
    WS_SAP_R,
    WS_SAP_PSI,
    WS_SAP_IN,
    WS_SOLVER,      // solver vectors
    WS_DFL,
    WS_CGNR,
    WS_MISC,
    WS_MISC2,
    WS_COARSE,
    WS_SOLVE_IO,
    WS_NET_PART,
    WS_NET_ACT,
    WS_NET_TGT,
    WS_NET_BATCH_T,
    WS_NET_FALLBACK,
    WS_HASEN,
    WS_PHI64,       // F64 preconditioner output converted into FP32 Krylov vectors
    WS_MD_OMEGA,    // per-site clover force weights (MD forces)
    WS_MD_SCRATCH,  // per-site partial sums (gauge action)
    WS_MD_FIELDS,   // pseudofermion force fields
    WS_MD_GRAD,     // MD gradient of the leapfrog step
};
lqcd_status ws_get(lqcd_ctx *c, int slot, size_t bytes, void **out);

// native element counts per site
size_t native_half_bytes(const lqcd_ctx *c, lqcd_prec p);   // one rhs, one parity
inline long native_half_units(const lqcd_ctx *c, lqcd_prec p)   // in 16-byte units
{
    return (long)(native_half_bytes(c, p) / 16);
}

// Launch whose CTAs may be set up while the kernel before it in the stream is
// still running (programmatic dependent launch); the kernel begins with
// after_previous(), which waits until that kernel has finished and its writes are
// visible.  It hides about 2 us per kernel: Dhat FP64 on 8^4 (four kernels) 28.7
// -> 19.3 us.  The CTAs set up early go to the SMs that come free first; where that
// spreads a kernel of about one wave unevenly it costs up to a third, so stencils
// (run_operator) and SAP sweeps choose.  The coarse solve's kernels are faster with it
// at every size timed (a deflated step of one field 0.68 at 8^4 to 0.93 at 48 x 24^3 of
// its time with plain launches), the canonical conversions at all but a few (calls of
// 0.8 to 1.03, one of 1.2, of their time with plain launches).  Kernels must let the
// next one be set up only after their own wait: signalled before it, the launches of
// a chain pile up on the SMs (43.6 us).  In captured graphs plain launches are faster
// (CGNR on 8^4: 6.97 against 7.97 ms).
// A launch that fails leaves its error for LQCD_LAUNCH_CHECK, as <<< >>> does.
template <class... KP, class... A>
inline void launch_pdl_smem(bool pdl, void (*kernel)(KP...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                            const A &...args)
{
    if (!pdl) {
        kernel<<<grid, block, smem, st>>>(args...);
        return;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cudaLaunchKernelEx(&cfg, kernel, static_cast<KP>(args)...);
}
template <class... KP, class... A>
inline void launch_pdl(bool pdl, void (*kernel)(KP...), dim3 grid, dim3 block, cudaStream_t st, const A &...args)
{
    launch_pdl_smem(pdl, kernel, grid, block, 0, st, args...);
}
__device__ __forceinline__ void after_previous()
{
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();   // the next kernel may be set up now, but no later one
}

// launch helpers
inline int div_up(long a, long b) { return (int)((a + b - 1) / b); }

// --------------------------------------------------------------- internals
// dirac
lqcd_status dirac_dhat(lqcd_ctx *c, lqcd_prec p, const void *in, void *out, void *tmp_o, int nrhs);
lqcd_status dirac_dhat_s(lqcd_ctx *c, lqcd_prec p, const void *in, long in_rs, void *out, long out_rs, void *tmp_o,
                         int nrhs);
lqcd_status dirac_D(lqcd_ctx *c, lqcd_prec p, const void *in, void *out, int nrhs);
lqcd_status dirac_hop_parity(lqcd_ctx *c, lqcd_prec p, int p_out, const void *in_other,
                             void *out, long in_rstride, long out_rstride, int nrhs);
// nhalf half fields; in_hs, out_hs: distance of consecutive ones in half fields
lqcd_status convert_native(lqcd_ctx *c, lqcd_prec from, lqcd_prec to, const void *in, void *out,
                           long nhalf, long in_hs = 1, long out_hs = 1);
lqcd_status pack_field(lqcd_ctx *c, lqcd_prec p, int nsub, const void *canon, void *native,
                       int nrhs, bool unpack);
// even_scale != 1: the even-site blocks of A (and so of A^-1) belong to
// even_scale * A_ee (the shifted operator of the Hasenbusch solve)
lqcd_status clover_build(lqcd_ctx *c, double kappa, double csw, double *ld_e, double *ld_o, double even_scale = 1.0);
lqcd_status clover_apply_native64(lqcd_ctx *c, int parity, int inverse, const double2 *in,
                                  double2 *out);

// blas (FP64 native vectors viewed as arrays of double; complex pairs)
lqcd_status blas_dot(lqcd_ctx *c, long n2, const double *a, const double *b, int k, long stride_a,
                     double *host_out);  // k dots <a_i, b>, host_out: 2k doubles
lqcd_status blas_norm2(lqcd_ctx *c, long n2, const double *a, double *host_out);
lqcd_status blas_axpy(lqcd_ctx *c, long n2, double ar, double ai, const double *x, double *y);
lqcd_status blas_scal(lqcd_ctx *c, long n2, double ar, double ai, double *y);
lqcd_status blas_copy(lqcd_ctx *c, long n2, const double *x, double *y);
lqcd_status blas_sub(lqcd_ctx *c, long n2, const double *x, const double *y, double *z);  // z = x - y
lqcd_status blas_multi_axpy(lqcd_ctx *c, long n2, int k, const double *coef_host, const double *X,
                            long stride, double *y, double sign);
lqcd_status bblas_dot(lqcd_ctx *c, long n2, int nrhs, const double *A, long sa, long fa, const double *B, long fb,
                      int k, double *host_out);
lqcd_status bblas_multi_axpy(lqcd_ctx *c, long n2, int nrhs, int k, const double *coef_host, const double *X,
                             long sa, long fa, double *y, long fy, double sign);
lqcd_status bblas_dot_dev(lqcd_ctx *c, long n2, int nrhs, const double *A, long sa, long fa, const double *B, long fb,
                          int k, double2 *out_dev);
lqcd_status bblas_multi_axpy_dev(lqcd_ctx *c, long n2, int nrhs, int k, const double2 *coef_dev, const double *X,
                                 long sa, long fa, double *y, long fy, double sign);
// GCR vectors.  nh: halves per vector (2: full fields, 1: their even halves);
// f*: distance of the right-hand sides.  dots land on the host as (re, im)
// pairs [r][i]; norm_rdot: [r][0] = |x_r|^2, [r][1] = <rho_r, x_r>.
lqcd_status bnorm_rdot64(lqcd_ctx *c, int nh, int nrhs, const double2 *x, long fx, const double2 *rho, long fr,
                         double *host_out);
lqcd_status brho_update64(lqcd_ctx *c, int nh, int nrhs, const double *cR_host, const double *sx_host, double2 *x,
                          long fx, double2 *rho, long fr);   // rho_r -= cR_r x_r; x_r *= sx_r
// rho_r = eta_r - w_r (w = NULL: eta_r), norms[r] = |rho_r|^2
lqcd_status bresidual64(lqcd_ctx *c, int nh, int nrhs, const double2 *eta, long fe, const double2 *w, long fw,
                        double2 *rho, long fr, double *norms);
// FP32 Krylov vectors: x, A, B, X, y are native F32 fields (float4, strides in
// float4), rho and psi native F64 fields (double2, strides in double2)
lqcd_status bdot32(lqcd_ctx *c, long n4, int nrhs, const float4 *A, long sa, long fa, const float4 *B, long fb, int k,
                   double *host_out);
lqcd_status bnorm_rdot32(lqcd_ctx *c, int nh, int nrhs, const float4 *x, long fx, const double2 *rho, long fr,
                         double *host_out);
lqcd_status bmulti_axpy32(lqcd_ctx *c, long n4, int nrhs, int k, const double *coef_host, const float4 *X, long sa,
                          long fa, float4 *y, long fy, double sign);
lqcd_status brho_update32(lqcd_ctx *c, int nh, int nrhs, const double *cR_host, const double *sx_host, float4 *x,
                          long fx, double2 *rho, long fr);   // rho_r -= cR_r x_r; x_r *= sx_r
lqcd_status bmulti_axpy_mixed(lqcd_ctx *c, int nh, int nrhs, int k, const double *coef_host, const float4 *X, long sa,
                              long fa, double2 *y, long fy);   // y_r += sum_i c_ri X_ir
lqcd_status blas_gamma5_native64(lqcd_ctx *c, long nhalf, const double2 *in, double2 *out);
lqcd_status blas_zero(lqcd_ctx *c, size_t bytes, void *p);

// even-odd CGNR (lqcd_cgnr.cu)
lqcd_status cgnr_native(lqcd_ctx *c, const double2 *eta, double2 *x, double tol, int nmx, lqcd_solve_info *info);

// sap
void sap_free_plans(lqcd_ctx *c);
lqcd_status sap_apply(lqcd_ctx *c, const lqcd_sap_params *sp, const void *eta_native,
                      void *psi_native, int nrhs = 1);
// batched operators over several lattices; hc: the batch's own context (stream,
// error text, launch counter); arenas hold the lattices' native full fields at
// offsets off[l] (in native spinor units of the precision)
struct DBatch;
lqcd_status dirac_batch_create(lqcd_ctx *hc, lqcd_ctx *const *ctx, int n, lqcd_prec p, const void *in, void *tmp,
                               void *out, const long *off, DBatch **out_b);
lqcd_status dirac_batch_dhat(lqcd_ctx *hc, DBatch *b, long shift, const int *active_dev);
void dirac_batch_free(DBatch *b);
struct SapBatch;
lqcd_status sap_batch_create(lqcd_ctx *hc, lqcd_ctx *const *ctx, int n, const lqcd_sap_params *sp, void *r,
                             void *psi, void *delta, const long *off, SapBatch **out_b);
lqcd_status sap_batch_apply(lqcd_ctx *hc, SapBatch *b, const void *eta, size_t bytes, const int *active_dev);
lqcd_status sap_batch_refresh(SapBatch *b, lqcd_ctx *const *ctx, int n, const int bs[4]);
void sap_batch_free(SapBatch *b);
void chrono_free(lqcd_ctx *c);
// learned preconditioner
void net_free(lqcd_ctx *c);
lqcd_status net_apply_native(lqcd_ctx *c, const double2 *rho, double2 *phi, int nrhs);
// deflation
void dfl_free(lqcd_ctx *c);
// smoother: SAP (net = false) or the network (net = true) after the deflation step
lqcd_status dfl_precond_native(lqcd_ctx *c, const lqcd_sap_params *sp, const double2 *rho,
                               double2 *phi, int nrhs, bool net = false);
lqcd_status dfl_precond_native32(lqcd_ctx *c, const lqcd_sap_params *sp, const double2 *rho, float4 *phi,
                                 int halves, int nrhs, bool *done);
