"""Conversions between FP64 and FP32 / FP16 fields in integer arithmetic: sites that
hold zeros, numbers below float's normal range and ordinary ones side by side (the
casts take over for such sites), seen through SAP in FP32 and FP16 against FP64 SAP
to the rounding of one application in that precision (1e-6, 3e-3)."""
import pytest

from paper_1011_0911_gb300 import lqcd, synth
from tests import util
from tests.gpu_util import links, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tol", [(lqcd.F32, 1e-6), (lqcd.F16S, 3e-3)], ids=["f32", "f16s"])
@pytest.mark.parametrize("scale", [0.0, 2.0 ** -130, -2.0 ** -1060, 1.0], ids=["zero", "subnormal32", "subnormal64", "normal"])
def test_mixed_magnitudes(prec, tol, scale):
    dims = (8, 4, 4, 8)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    ctx = lqcd.Context(dims)
    ctx.set_gauge(to_gpu(links(dims, 5)))
    ctx.clover_invert(0.1355, 1.9)
    eta = synth.gaussian_spinor(V, 81).reshape(V, 12)
    eta[::3, 1::2] *= scale      # within a site
    eta[1::5] *= scale           # whole sites
    eta = to_gpu(eta.reshape(V, 4, 3))
    ref = ctx.sap(eta, ncy=2, nmr=3, prec=lqcd.F64).cpu().numpy()
    out = ctx.sap(eta, ncy=2, nmr=3, prec=prec).cpu().numpy()
    assert util.relerr(out, ref) < tol
