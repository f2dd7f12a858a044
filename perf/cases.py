"""What is timed of this library, and how its results are checked.

Every case is one call, or one short run of calls, that a program working on a two-flavour Wilson-clover HMC makes
through the Python binding (paper_1011_0911_gb300.lqcd): operator applications, the Schwarz preconditioner, the
solvers, the subspace build, the force terms, the learned preconditioner.  Lattices, quark masses and solver parameters
are those of this repository's benchmark, tests and workloads.  Links are random SU(3) matrices of plaquette 0.55,
sources and momenta are Gaussian, all made from the seed on the GPU.

exact() recomputes the results with plain torch in 64 bits (class Ref), from the definitions in include/lqcd.h.
"""
import functools
import math

import numpy as np
import torch

from paper_1011_0911_gb300 import lqcd, synth

PREC = {"f64": lqcd.F64, "f32": lqcd.F32, "f16s": lqcd.F16S, "bf16": lqcd.BF16}
CSW = 1.9
BETA = 5.3
NET_CHANS = (1, 2, 2, 1)
BATCH_SIZES = ((8, 8, 8, 8), (16, 16, 16, 16), (24, 12, 12, 12), (32, 16, 16, 16))


def _case(kind, dims, kappa, **kw):
    return dict(kind=kind, T=dims[0], L1=dims[1], L2=dims[2], L3=dims[3], kappa=kappa, **kw)


def listed():
    return [
        # the smallest call: one FP64 Dhat on 8^4 (tests of an HMC, small-volume runs), canonical fields
        dict(name="dhat_f64_8x8", **_case("dhat", (8, 8, 8, 8), 0.1355, prec="f64", nrhs=1, native=False)),
        # the benchmark's step: FP32 Dhat on the 12 spin-colour sources of the production lattice, resident fields
        dict(name="dhat_f32_48x24_n12", **_case("dhat", (48, 24, 24, 24), 0.13625, prec="f32", nrhs=12, native=True)),
        # the FP64 operator at the production size: every residual check, restart and reversibility test is one
        dict(name="dhat_f64_48x24", **_case("dhat", (48, 24, 24, 24), 0.13625, prec="f64", nrhs=1, native=False)),
        # D on a lattice whose extents are no powers of two, an odd number of fields, canonical FP32
        dict(name="d_f32_28x12_n5", **_case("d", (28, 12, 10, 14), 0.1355, prec="f32", nrhs=5)),
        # plain even-odd CG on the normal equation, 8^4: launches, reductions and host waits
        dict(name="cgnr_f64_8x8", **_case("solve", (8, 8, 8, 8), 0.1355, solver="cgnr", sap_prec="f64", inner="f64",
                                          krylov="f64", nrhs=1)),
        # one application of the Schwarz preconditioner with the default parameters (FP64, 4 cycles x 5 MinRes steps)
        dict(name="sap_f64_32x16", **_case("sap", (32, 16, 16, 16), 0.1357, prec="f64", ncy=4, nmr=5)),
        # SAP-GCR for one source, FP32 preconditioner and stencil inside the FP64 GCR
        dict(name="solve_f32_32x16", **_case("solve", (32, 16, 16, 16), 0.1357, solver="sap", sap_prec="f32",
                                             inner="f32", krylov="f64", nrhs=1)),
        # time to solution at the production size: subspace build and 12 sources, the benchmark's fastest precisions
        dict(name="tts_48x24_n12", **_case("tts", (48, 24, 24, 24), 0.13625, nrhs=12, Ns=20)),
        # 16 lattices of four sizes solved together
        dict(name="batch_uneven_16", kind="batch", count=16, pick=0),
        # what an MD step does with a new gauge field besides its solves: load it, build and invert the clover term,
        # and the three force terms
        dict(name="md_force_32x16", **_case("force", (32, 16, 16, 16), 0.1357)),
        # the block inversions of the DD-HMC, blocks of 6^2 x 12^2
        dict(name="block_48x24", **_case("block", (48, 24, 24, 24), 0.13625, b0=6, b1=6, b2=12, b3=12)),
        # the learned preconditioner applied to four fields of its training lattice
        dict(name="net_bf16_32x16_n4", **_case("net", (32, 16, 16, 16), 0.1363, prec="bf16", nrhs=4)),
    ]


# ------------------------------------------------------------------ drawn cases
def _extents(rng, step, lo, hi, least):
    """Four extents, multiples of step, of a volume spread over the logarithm of lo..hi."""
    target = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    side = (target / 2) ** 0.25
    L = [min(24, max(least, step * round(side * rng.uniform(0.7, 1.4) / step))) for _ in range(3)]
    t = step * round(target / (L[0] * L[1] * L[2]) / step)
    t = min(48, max(least, t))
    while t > least and t * L[0] * L[1] * L[2] > hi:
        t -= step
    return (t, L[0], L[1], L[2])


def draw(rng):
    kind = rng.choice(("dhat", "dhat", "d", "cgnr", "sap", "solve", "solve", "tts", "batch", "force", "block", "net"))
    kappa = round(rng.uniform(0.1350, 0.1362), 5)
    full = 48 * 24 ** 3
    if kind in ("dhat", "d"):
        prec = rng.choice(("f64", "f32", "f32", "f16s"))
        dims = _extents(rng, 2, 4096, full, 4)
        vol = dims[0] * dims[1] * dims[2] * dims[3]
        n = rng.choice([k for k in (1, 2, 3, 4, 5, 7, 12) if k * vol <= 12 * full and (prec != "f64" or k <= 4)])
        if kind == "d":
            return _case("d", dims, kappa, prec=prec, nrhs=n)
        return _case("dhat", dims, kappa, prec=prec, nrhs=n, native=rng.random() < 0.5 and prec != "f16s")
    if kind == "cgnr":
        return _case("solve", _extents(rng, 2, 2048, 32768, 4), kappa, solver="cgnr", sap_prec="f64", inner="f64",
                     krylov="f64", nrhs=1)
    if kind == "sap":
        ncy, nmr = rng.choice(((4, 5), (1, 4), (2, 8), (6, 4)))
        return _case("sap", _extents(rng, 4, 4096, 32 * 16 ** 3, 8), kappa, prec="f64", ncy=ncy, nmr=nmr)
    if kind == "solve":
        p = rng.choice(("f64", "f32", "f32", "f16s"))
        dims = _extents(rng, 4, 4096, 32 * 16 ** 3 // (2 if p == "f64" else 1), 8)
        inner = "f64" if p == "f64" else "f32"
        return _case("solve", dims, kappa, solver="sap", sap_prec=p, inner=inner,
                     krylov=rng.choice(("f64", "f32")) if inner == "f32" else "f64",
                     nrhs=1 if p == "f64" else rng.choice((1, 2, 3)))
    if kind == "tts":
        return _case("tts", _extents(rng, 8, 32768, 32 * 16 ** 3, 8), kappa, nrhs=rng.choice((1, 4, 7, 12)),
                     Ns=rng.choice((12, 16, 20)))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(2, 12), pick=rng.randint(1, 1000))
    if kind == "force":
        return _case("force", _extents(rng, 2, 4096, 32 * 16 ** 3, 4), kappa)
    if kind == "block":
        b = [rng.choice((4, 6, 8)) for _ in range(4)]
        dims = tuple(b[i] * rng.choice((2, 3) if i else (2, 4)) for i in range(4))
        return _case("block", dims, kappa, b0=b[0], b1=b[1], b2=b[2], b3=b[3])
    return _case("net", _extents(rng, 2, 4096, 32 * 16 ** 3, 4), kappa, prec=rng.choice(("bf16", "bf16", "f32")),
                 nrhs=rng.choice((1, 3, 4)))


# ------------------------------------------------------------------ inputs
def _dims(case):
    return (case["T"], case["L1"], case["L2"], case["L3"])


def _gen(seed, stream):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 64 + stream) % (1 << 62))


def _gauss(seed, stream, shape):
    return torch.randn(shape, dtype=torch.complex128, device="cuda", generator=_gen(seed, stream)) * math.sqrt(2.0)


@functools.lru_cache(maxsize=None)
def _gell_mann():
    return torch.from_numpy(synth.gell_mann()).cuda()


def _links(dims, seed, stream=1):
    """U = exp(i eps H), H = sum_a h_a lambda_a / 2, h_a normal, eps for a plaquette of 0.55; SU(3) to rounding."""
    n = 4 * dims[0] * dims[1] * dims[2] * dims[3]
    h = torch.randn((n, 8), dtype=torch.float64, device="cuda", generator=_gen(seed, stream))
    X = (1j * synth.tuned_eps() / 2 / 8) * torch.einsum("na,aij->nij", h.to(torch.complex128), _gell_mann())
    U = torch.eye(3, dtype=torch.complex128, device="cuda") + X / 8
    for k in range(7, 0, -1):   # Horner form of the exponential series of X, squared three times
        U = torch.eye(3, dtype=torch.complex128, device="cuda") + (X @ U) / k
    for _ in range(3):
        U = U @ U
    a = U[:, 0] / U[:, 0].abs().square().sum(1, keepdim=True).sqrt()
    b = U[:, 1] - (a.conj() * U[:, 1]).sum(1, keepdim=True) * a
    b = b / b.abs().square().sum(1, keepdim=True).sqrt()
    c = torch.linalg.cross(a, b).conj()
    return torch.stack((a, b, c), 1).reshape(n // 4, 4, 3, 3).contiguous()


def _net_weights(seed):
    """0.7 on the identity path plus small noise: what the network is trained from."""
    rng = np.random.default_rng(int(seed))
    out = []
    for ci, co in zip(NET_CHANS[:-1], NET_CHANS[1:]):
        w = 0.02 * (rng.standard_normal((co, ci, 9, 4, 4)) + 1j * rng.standard_normal((co, ci, 9, 4, 4)))
        w[0, 0, 0] += 0.7 * np.eye(4)
        out.append(w.reshape(-1))
    return np.concatenate(out).astype(np.complex64)


def _batch(case):
    """(extents, kappa) of every lattice of a batch."""
    rng = np.random.default_rng(case["pick"])
    picks = rng.integers(0, len(BATCH_SIZES), case["count"])
    kappas = rng.uniform(0.1350, 0.1360, case["count"])
    return [(BATCH_SIZES[int(i)], float(k)) for i, k in zip(picks, kappas)]


def _inputs(case, seed):
    """The host program's data for a case, without the library: links, sources, momenta, weights."""
    kind = case["kind"]
    if kind == "batch":
        lat = _batch(case)
        return {"U": [_links(d, seed, 100 + i) for i, (d, _) in enumerate(lat)],
                "eta": [_gauss(seed, 200 + i, (d[0] * d[1] * d[2] * d[3] // 2, 4, 3)) for i, (d, _) in enumerate(lat)]}
    dims = _dims(case)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    d = {"U": _links(dims, seed)}
    if kind in ("dhat", "d"):
        x = _gauss(seed, 2, (case["nrhs"], V // 2 if kind == "dhat" else V, 4, 3))
        d["x"] = x if case["prec"] == "f64" else x.to(torch.complex64)
    elif kind in ("solve", "tts"):
        d["eta"] = _gauss(seed, 2, (case["nrhs"], V // 2, 4, 3))
        if kind == "tts":
            d["v0"] = _gauss(seed, 3, (case["Ns"], V, 4, 3))
    elif kind == "block":
        d["eta"] = _gauss(seed, 2, (V // 2, 4, 3))
    elif kind == "sap":
        d["eta"] = _gauss(seed, 2, (V, 4, 3))
    elif kind == "force":
        d["X"], d["Y"] = _gauss(seed, 2, (V, 4, 3)), _gauss(seed, 3, (V, 4, 3))
    elif kind == "net":
        d["x"] = _gauss(seed, 2, (case["nrhs"], V, 4, 3))
        d["W"] = _net_weights(seed)
    return d


def _context(dims, U, kappa):
    ctx = lqcd.Context(dims)
    ctx.set_gauge(U)
    ctx.clover_invert(kappa, CSW)
    return ctx


def prepare(case, seed):
    s = dict(_inputs(case, seed), case=case)
    kind = case["kind"]
    if kind == "batch":
        ctxs = [_context(d, U, k) for (d, k), U in zip(_batch(case), s.pop("U"))]
        s["batch"] = lqcd.Batch(ctxs, nkv=16, nmx=4096, tol=1e-12, sap_prec=lqcd.F16S)
        return s
    s["ctx"] = _context(_dims(case), s["U"], case["kappa"])
    if kind != "force":
        del s["U"]
    if kind == "dhat" and case["native"]:
        p = PREC[case["prec"]]
        s["x"] = s["ctx"].pack(s["x"], p, 1)
        s["out"] = s["ctx"].native_empty(p, 1, case["nrhs"])
    elif kind == "net":
        s["ctx"].net_set(NET_CHANS, s.pop("W"), act=PREC[case["prec"]])
    return s


def run(s):
    case, ctx = s["case"], s.get("ctx")
    kind = case["kind"]
    if kind == "dhat":
        p = PREC[case["prec"]]
        if not case["native"]:
            return ctx.apply_Dhat(s["x"], p)
        ctx.apply_Dhat_native(s["x"], s["out"], p, case["nrhs"])
        return s["out"].view(torch.float64 if case["prec"] == "f64" else torch.float32)
    if kind == "d":
        return ctx.apply_D(s["x"], PREC[case["prec"]])
    if kind == "sap":
        return ctx.sap(s["eta"], ncy=case["ncy"], nmr=case["nmr"], prec=PREC[case["prec"]])
    if kind == "solve":
        sid = lqcd.SOLVER_CGNR if case["solver"] == "cgnr" else lqcd.SOLVER_SAP_GCR
        psi, _, _ = ctx.solve_dhat(s["eta"], solver=sid, tol=1e-12, nmx=20000, sap_prec=PREC[case["sap_prec"]],
                                   inner=PREC[case["inner"]], krylov=PREC[case["krylov"]])
        return psi
    if kind == "tts":
        ctx.dfl_build(s["v0"], ninv=6, ncy=6, nmr=4, prec=lqcd.F32, coarse_tol=1e-2, coarse_nkv=32, coarse_nmx=32,
                      coarse_prec=lqcd.F32, build_sap_prec=lqcd.F16S, coarse_eo=True)
        psi, _, _ = ctx.solve_dhat(s["eta"], solver=lqcd.SOLVER_DFL_SAP_GCR, tol=1e-12, sap_prec=lqcd.F16S,
                                   inner=lqcd.F32, krylov=lqcd.F32, ncy=1, nmr=4)
        return [psi[k] for k in range(case["nrhs"])]
    if kind == "batch":
        return s["batch"].solve_dhat(s["eta"], check=True)[0]
    if kind == "force":
        ctx.set_gauge(s["U"])
        ld = ctx.clover_invert(case["kappa"], CSW)
        return {"logdet": ld, "dD": ctx.force_dD(s["X"], s["Y"]), "det": ctx.force_logdet(1),
                "gauge": ctx.force_gauge(BETA)}
    if kind == "block":
        return ctx.block_solve(s["eta"], (case["b0"], case["b1"], case["b2"], case["b3"]), tol=1e-12)[0]
    return ctx.net_apply(s["x"])


def work(case):
    """One pass: the bytes of its operands, read or written once, and the operations of its method: 3672 per even site
    for one Dhat, 1848 per site for one D, times a usual number of applications in the solvers."""
    if case["kind"] == "batch":
        V = sum(d[0] * d[1] * d[2] * d[3] for d, _ in _batch(case))
        return {"bytes": V * (8 * 72.0 + 4 * 36 + 2 * 96), "flops": V * 1848.0 * 70 * 25}
    dims = _dims(case)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    kind, n = case["kind"], case.get("nrhs", 1)
    word = {"f64": 8, "f32": 4, "f16s": 2}.get(case.get("prec", "f64"), 8)
    # words a site of the links (two rows where they are rebuilt) and of the clover term
    op = V * word * ((72 if word == 8 else 48) + 72)
    if kind == "dhat":
        return {"bytes": op + n * V / 2 * 48 * word, "flops": n * V / 2 * 3672.0}
    if kind == "d":
        return {"bytes": op + n * V * 48 * max(word, 4), "flops": n * V * 1848.0}
    if kind == "sap":
        return {"bytes": op + V * 48 * 8, "flops": V * 1848.0 * case["ncy"] * (case["nmr"] + 2)}
    if kind == "solve":
        its = 260 if case["solver"] == "cgnr" else 60 * 25
        return {"bytes": op + n * V / 2 * 48 * 8, "flops": n * V / 2 * 3672.0 * its}
    if kind == "tts":
        build, solve = case["Ns"] * 6 * 6 * 6, 32 * 9 * n
        return {"bytes": V * 8.0 * (144 + 24 * case["Ns"] + 24 * n), "flops": V * 1848.0 * (build + solve)}
    if kind == "force":
        # clover term: 24 leaves of 3 products; forces: 6 staples a link, 8 products with the clover weights each
        return {"bytes": V * 8.0 * (72 + 2 * 72 + 48 + 3 * 32), "flops": V * 198.0 * (24 * 3 + 4 * 6 * (8 + 2))}
    if kind == "block":
        return {"bytes": op + V / 2 * 48 * 8, "flops": V / 2 * 3672.0 * 90}
    return {"bytes": V * (4.0 * 48 + n * 48 * 8), "flops": n * V * (40 * 4 * 66 + 6 * 9 * 16 * 8 * 3.0)}


# ------------------------------------------------------------------ the same in 64 bits
class Ref:
    """The Wilson-clover operator on a grid, complex128.  Fields are (T, L1, L2, L3, colour 3, spin 4, n)."""

    def __init__(self, dims, U, kappa, clover=True):
        self.dims, self.V = dims, U.shape[0]
        self.U = U.reshape(*dims, 4, 3, 3)
        x = torch.stack(torch.meshgrid(*[torch.arange(L, device=U.device) for L in dims], indexing="ij"))
        self.x, self.parity = x, (x.sum(0) & 1)
        self.even = (self.parity == 0).reshape(-1).nonzero()[:, 0]
        s = torch.zeros((3, 2, 2), dtype=torch.complex128, device=U.device)
        s[0, 0, 1] = s[0, 1, 0] = 1
        s[1, 0, 1], s[1, 1, 0] = -1j, 1j
        s[2, 0, 0], s[2, 1, 1] = 1, -1
        e = torch.cat((-torch.eye(2, dtype=torch.complex128, device=U.device)[None], -1j * s))
        g = torch.zeros((4, 4, 4), dtype=torch.complex128, device=U.device)
        g[:, :2, 2:], g[:, 2:, :2] = e, e.conj().transpose(1, 2)
        self.gamma = g
        self.g5 = torch.tensor([1.0, 1, -1, -1], device=U.device, dtype=torch.float64)[:, None]
        perm = g.abs().argmax(2)
        self.perm = [p for p in perm]
        self.phase = [g[m].gather(1, perm[m][:, None]) for m in range(4)]
        # time-boundary signs of the forward and the backward hop in direction 0
        one = torch.ones(dims, dtype=torch.float64, device=U.device)
        self.sign = [torch.where(x[0] == dims[0] - 1, -one, one), torch.where(x[0] == 0, -one, one)]
        self.mask = None
        if clover:
            self.A = self.clover(self.U, kappa)
            self.Ai = torch.linalg.inv(self.A)

    @staticmethod
    def at(f, mu, d):
        return torch.roll(f, -d, mu)

    def clover(self, U, kappa):
        """A(x) as 12 x 12 matrices, index 4 colour + spin."""
        A = (1 / (2 * kappa)) * torch.eye(12, dtype=torch.complex128, device=U.device)
        A = A.expand(*self.dims, 12, 12).clone()
        for m in range(4):
            for n in range(m + 1, 4):
                Q = self.leaves(U[..., m, :, :], U[..., n, :, :], m, n)
                F = (Q - Q.conj().transpose(-1, -2)) / 8
                sg = 0.5j * (self.gamma[m] @ self.gamma[n] - self.gamma[n] @ self.gamma[m])
                A = A + CSW * 0.5j * torch.einsum("...ij,st->...isjt", F, sg).reshape(*self.dims, 12, 12)
        return A

    def leaves(self, a, b, m, n):
        """Sum of the four plaquette leaves at x in the plane (m, n)."""
        at = self.at
        dag = lambda u: u.conj().transpose(-1, -2)   # noqa: E731
        am, bn = at(a, m, -1), at(b, n, -1)          # U_m(x-m), U_n(x-n)
        bm_n, am_n = at(at(b, m, -1), n, -1), at(am, n, -1)
        return (a @ at(b, m, 1) @ dag(at(a, n, 1)) @ dag(b)
                + b @ dag(at(am, n, 1)) @ dag(at(b, m, -1)) @ am
                + dag(am) @ dag(bm_n) @ am_n @ bn
                + dag(bn) @ at(a, n, -1) @ at(bn, m, 1) @ dag(a))

    def blocks(self, bs):
        """Keep only the hops inside blocks of these extents."""
        self.mask = []
        for m in range(4):
            for d in (1, -1):
                y = (self.x[m] + d) % self.dims[m]
                self.mask.append((y // bs[m] == self.x[m] // bs[m]).to(torch.float64)[..., None, None, None])

    def hop(self, psi, U=None, mask=None):
        """H psi = -1/2 sum of the eight hops."""
        U = self.U if U is None else U
        n = psi.shape[-1]
        out = 0
        for m in range(4):
            gp = psi[..., self.perm[m], :] * self.phase[m]
            f, b = psi - gp, psi + gp
            u = U[..., m, :, :]
            f = self.at(f, m, 1).reshape(*self.dims, 3, 4 * n)
            f = (u @ f).reshape(psi.shape)
            b = self.at(u.conj().transpose(-1, -2) @ b.reshape(*self.dims, 3, 4 * n), m, -1).reshape(psi.shape)
            if m == 0:
                f, b = f * self.sign[0][..., None, None, None], b * self.sign[1][..., None, None, None]
            if mask is not None:
                f, b = f * mask[2 * m], b * mask[2 * m + 1]
            out = out + f + b
        return -0.5 * out

    def site(self, A, psi):
        return (A @ psi.reshape(*self.dims, 12, -1)).reshape(psi.shape)

    def on(self, p, psi):
        return psi * (self.parity == p)[..., None, None, None]

    def D(self, psi):
        return self.site(self.A, psi) + self.hop(psi)

    def Dhat(self, psi):
        """Even field in, even field out (zero on odd sites); inside blocks where these are set."""
        t = self.site(self.Ai, self.hop(psi, mask=self.mask))
        return self.site(self.A, psi) - self.hop(t, mask=self.mask)

    def full(self, c):
        """canonical (n, V, 4, 3) -> grid"""
        return c.to(torch.complex128).permute(1, 3, 2, 0).reshape(*self.dims, 3, 4, -1)

    def canon(self, f):
        return f.reshape(self.V, 3, 4, -1).permute(3, 0, 2, 1)

    def from_even(self, c):
        f = torch.zeros((c.shape[0], self.V, 4, 3), dtype=torch.complex128, device=c.device)
        f[:, self.even] = c.to(torch.complex128)
        return self.full(f)

    def to_even(self, f):
        return self.canon(f)[:, self.even]

    def solve(self, eta, tol=2e-15, nmx=3000):
        """Dhat psi = eta by CG on the normal equation, to rounding, all fields together."""
        dot = lambda a, b: (a.conj() * b).real.flatten(0, -2).sum(0)   # noqa: E731
        dagger = lambda v: self.g5 * self.Dhat(self.g5 * v)            # noqa: E731
        x, e2 = torch.zeros_like(eta), dot(eta, eta)
        for _ in range(3):   # each pass starts from the recomputed residual
            r = eta - self.Dhat(x)
            z = dagger(r)
            p, zz = z.clone(), dot(z, z)
            for k in range(nmx):
                w = self.Dhat(p)
                a = zz / dot(w, w).clamp_min(1e-300)
                x, r = x + a * p, r - a * w
                if k % 20 == 19 and bool((dot(r, r) <= (tol * tol) * e2).all()):
                    break
                z = dagger(r)
                z2 = dot(z, z)
                p, zz = z + (z2 / zz.clamp_min(1e-300)) * p, z2
        return x

    def sap(self, eta, bs, ncy, nmr):
        """The Schwarz alternating procedure: block colour after block colour, MinRes on every block's Dhat."""
        self.blocks(bs)
        nb = [L // b for L, b in zip(self.dims, bs)]
        col = sum(self.x[m] // bs[m] for m in range(4)) & 1

        def bsum(v):   # per-block sum of a site quantity, spread back over the block's sites
            s = v.flatten(4).sum(-1).reshape(nb[0], bs[0], nb[1], bs[1], nb[2], bs[2], nb[3], bs[3])
            s = s.sum((1, 3, 5, 7), keepdim=True).expand(nb[0], bs[0], nb[1], bs[1], nb[2], bs[2], nb[3], bs[3])
            return s.reshape(*self.dims)[..., None, None, None]

        psi, r = torch.zeros_like(eta), eta
        for _ in range(ncy):
            for c in range(2):
                ro, re = self.on(1, r), self.on(0, r)
                rho = re - self.hop(self.site(self.Ai, ro), mask=self.mask)
                chi = torch.zeros_like(rho)
                for _ in range(nmr):
                    p = self.Dhat(rho)
                    pp = bsum((p.conj() * p).real)
                    a = torch.where(pp > 0, bsum(p.conj() * rho) / pp.clamp_min(1e-300), 0)
                    chi, rho = chi + a * rho, rho - a * p
                chi = chi + self.site(self.Ai, ro - self.hop(chi, mask=self.mask))
                psi = psi + chi * (col == c)[..., None, None, None]
                r = eta - self.D(psi)
        return psi

    def forces(self, kappa, X, Y):
        """Gradients at eps = 0 of Re <Y, D X>, log|det A_oo| and the gauge action under U -> exp(eps_a T_a) U."""
        T = 0.5j * _gell_mann()
        eps = torch.zeros((*self.dims, 4, 8), dtype=torch.float64, device=self.U.device, requires_grad=True)
        step = torch.einsum("...a,aij->...ij", eps.to(torch.complex128), T)
        U = self.U + step @ self.U
        A = self.clover(U, kappa)
        f = (Y.conj() * (self.site(A, X) + self.hop(X, U))).real.sum()
        odd = A.reshape(self.V, 12, 12)[(self.parity == 1).reshape(-1)]
        ld = torch.linalg.slogdet(odd)[1].sum()
        S = 0
        for m in range(4):
            for n in range(m + 1, 4):
                a, b = U[..., m, :, :], U[..., n, :, :]
                P = a @ self.at(b, m, 1) @ self.at(a, n, 1).conj().transpose(-1, -2) @ b.conj().transpose(-1, -2)
                S = S + BETA * (1 - P.diagonal(dim1=-2, dim2=-1).sum(-1).real / 3).sum()
        return [torch.autograd.grad(v, eps, retain_graph=True)[0].reshape(self.V, 4, 8) for v in (f, ld, S)]

    def net(self, x, W):
        n, W, y = x.shape[-1], torch.from_numpy(W.astype(np.complex128)).cuda(), [x]
        at = 0
        for ci, co in zip(NET_CHANS[:-1], NET_CHANS[1:]):
            w = W[at:at + co * ci * 144].reshape(co, ci, 9, 4, 4)
            at += co * ci * 144
            out = [0] * co
            for i in range(ci):
                tr = [y[i]]
                for m in range(4):
                    u = self.U[..., m, :, :]
                    f = (u @ self.at(y[i], m, 1).reshape(*self.dims, 3, 4 * n)).reshape(y[i].shape)
                    b = self.at(u.conj().transpose(-1, -2) @ y[i].reshape(*self.dims, 3, 4 * n), m, -1).reshape(
                        y[i].shape)
                    if m == 0:
                        f, b = f * self.sign[0][..., None, None, None], b * self.sign[1][..., None, None, None]
                    tr += [f, b]
                for o in range(co):
                    out[o] = out[o] + sum(torch.einsum("st,...ctn->...csn", w[o, i, d], tr[d]) for d in range(9))
            y = out
        return y[0]


def exact(case, seed):
    s = _inputs(case, seed)
    kind = case["kind"]
    if kind == "batch":
        out = []
        for (dims, kappa), U, eta in zip(_batch(case), s["U"], s["eta"]):
            R = Ref(dims, U, kappa)
            out.append(R.to_even(R.solve(R.from_even(eta[None])))[0] if len(out) < 4 else None)
        return out
    dims = _dims(case)
    R = Ref(dims, s["U"], case["kappa"], clover=kind != "net")
    if kind == "dhat":
        fields = [R.to_even(R.Dhat(R.from_even(s["x"][k:k + 1]))) for k in range(case["nrhs"])]
        out = torch.cat(fields)
        if not case["native"]:
            return out
        w = 1 if case["prec"] == "f64" else 2   # complex numbers in a 16-byte word of the resident layout
        out = torch.view_as_real(out.reshape(case["nrhs"], -1, 12 // w, w)).flatten(3)
        return out.transpose(1, 2).reshape(-1)
    if kind == "d":
        return torch.cat([R.canon(R.D(R.full(s["x"][k:k + 1]))) for k in range(case["nrhs"])])
    if kind == "sap":
        return R.canon(R.sap(R.full(s["eta"][None]), (4, 4, 4, 4), case["ncy"], case["nmr"]))[0]
    if kind == "solve":
        return R.to_even(R.solve(R.from_even(s["eta"])))
    if kind == "tts":
        if R.V > 32 * 16 ** 3:   # about a minute
            return None
        return [R.to_even(R.solve(R.from_even(s["eta"][:1])))[0]] + [None] * (case["nrhs"] - 1)
    if kind == "block":
        R.blocks((case["b0"], case["b1"], case["b2"], case["b3"]))
        return R.to_even(R.solve(R.from_even(s["eta"][None])))[0]
    if kind == "force":
        ld = torch.linalg.slogdet(R.A.reshape(R.V, 12, 12))[1]
        odd = (R.parity == 1).reshape(-1)
        g = R.forces(case["kappa"], R.full(s["X"][None]), R.full(s["Y"][None]))
        return {"logdet": (float(ld[~odd].sum()), float(ld[odd].sum())), "dD": g[0], "det": g[1], "gauge": g[2]}
    return R.canon(R.net(R.full(s["x"]), s["W"]))
