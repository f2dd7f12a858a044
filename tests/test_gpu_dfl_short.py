"""The deflated preconditioner with an FP32 subspace and short SAP fields (one pass
each for the residual and the sum) against its parts through their own entry points,
u = Pi A^-1 Pi^dag rho, u + M_sap (rho - D u): the same values up to the rounding of
one SAP application in its precision (1e-6, 3e-3).  Two block shapes: two threads a
site in the expansion, and the general kernel (blocks of 96 sites)."""
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests import util
from tests.gpu_util import links, to_gpu

pytestmark = pytest.mark.gpu

DIMS = (8, 4, 12, 8)


@pytest.mark.parametrize("bs", [(4, 4, 4, 4), (2, 4, 6, 2)], ids=["4x4x4x4", "2x4x6x2"])
@pytest.mark.parametrize("prec,tol", [(lqcd.F32, 1e-6), (lqcd.F16S, 3e-3)], ids=["f32", "f16s"])
def test_matches_its_parts(bs, prec, tol):
    V = DIMS[0] * DIMS[1] * DIMS[2] * DIMS[3]
    ctx = lqcd.Context(DIMS)
    ctx.set_gauge(to_gpu(links(DIMS, 4)))
    ctx.clover_invert(0.1355, 1.9)
    v0 = synth.gaussian_spinor(5 * V, 71).reshape(5, V, 4, 3)
    ctx.dfl_build(to_gpu(v0), bs=bs, ninv=2, ncy=2, nmr=4, prec=lqcd.F32, coarse_tol=1e-10)
    rho = to_gpu(synth.gaussian_spinor(V, 72)).view(V, 4, 3)
    u = ctx.dfl_expand(ctx.dfl_coarse_solve(ctx.dfl_project(rho))[0])
    w = rho - ctx.apply_D(u, prec=prec).to(torch.complex128).view_as(rho)
    ref = u + ctx.sap(w, ncy=3, nmr=4, prec=prec).view_as(rho)
    out = ctx.dfl_precond(rho, ncy=3, nmr=4, prec=prec)
    assert util.relerr(out.cpu().numpy(), ref.cpu().numpy()) < tol


@pytest.mark.parametrize("dims,bs,Ns", [((8, 4, 12, 8), (4, 4, 4, 4), 5), ((8, 4, 12, 8), (2, 4, 6, 2), 3),
                                        ((4, 4, 8, 16), (2, 2, 2, 16), 8), ((4, 8, 4, 4), (4, 8, 4, 4), 9)],
                         ids=["wrapped", "faces-not-whole-warps", "long-block", "one-block"])
def test_little_operator_is_the_projected_operator(dims, bs, Ns):
    """A = Pi^dag D Pi of an FP32 subspace, column groups partly filled: applied to a
    vector it agrees with the three parts in turn to the FP32 rounding of sums over a
    block (1e-5, as for the operator against the oracle)."""
    V = dims[0] * dims[1] * dims[2] * dims[3]
    ctx = lqcd.Context(dims)
    ctx.set_gauge(to_gpu(links(dims, 6)))
    ctx.clover_invert(0.1355, 1.9)
    v0 = synth.gaussian_spinor(Ns * V, 73).reshape(Ns, V, 4, 3)
    ctx.dfl_build(to_gpu(v0), bs=bs, ninv=1, ncy=2, nmr=4, prec=lqcd.F32, coarse_tol=1e-8)
    n = ctx.nblk * Ns
    c = to_gpu(synth.gaussian_spinor(n, 74).reshape(-1)[:n].copy())
    ref = ctx.dfl_project(ctx.apply_D(ctx.dfl_expand(c)))
    assert util.relerr(ctx.dfl_little_apply(c).cpu().numpy(), ref.cpu().numpy()) < 1e-5
