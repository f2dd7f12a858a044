"""The block-ordered operator copy of the resident SAP kernel: after a new gauge
field or clover term, for two block shapes of one context, and in a batch made
before the change, the result is that of a fresh context, bit for bit."""
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import links, to_gpu

pytestmark = pytest.mark.gpu

DIMS = (8, 4, 12, 4)


def fresh(U, kappa):
    ctx = lqcd.Context(DIMS)
    ctx.set_gauge(to_gpu(U))
    ctx.clover_invert(kappa, 1.9)
    return ctx


@pytest.mark.parametrize("prec", [lqcd.F32, lqcd.F16S], ids=["f32", "f16s"])
def test_copy_follows_the_operator(prec):
    eta = to_gpu(synth.gaussian_spinor(8 * 4 * 12 * 4, 51))
    ctx = fresh(links(DIMS, 0), 0.1355)
    shapes = [(4, 4, 4, 4), (4, 2, 4, 2), (2, 4, 6, 4)]
    for U, kappa in ((links(DIMS, 0), 0.1355), (links(DIMS, 0), 0.1340), (links(DIMS, 1), 0.1340)):
        ctx.set_gauge(to_gpu(U))
        ctx.clover_invert(kappa, 1.9)
        ref = fresh(U, kappa)
        for bs in shapes:
            kw = dict(bs=bs, ncy=2, nmr=3, prec=prec)
            assert torch.equal(ctx.sap(eta, **kw), ref.sap(eta, **kw)), (kappa, bs)


def test_batch_made_before_the_change():
    ctx = fresh(links(DIMS, 0), 0.1355)
    B = lqcd.Batch([ctx], tol=1e-10)
    e = to_gpu(synth.gaussian_spinor(8 * 4 * 12 * 2, 52))
    B.solve_dhat([e], check=True)
    ctx.set_gauge(to_gpu(links(DIMS, 1)))
    ctx.clover_invert(0.1350, 1.9)
    psi, info, st = B.solve_dhat([e], check=True)
    ref = lqcd.Batch([fresh(links(DIMS, 1), 0.1350)], tol=1e-10)
    rpsi, rinfo, rst = ref.solve_dhat([e], check=True)
    assert info[0]["iters"] == rinfo[0]["iters"]
    assert torch.equal(psi[0], rpsi[0])
