"""The GCR on even fields: several right-hand sides with strided halves, in every
storage of its Krylov vectors, from zero and from a guess; one source is zero."""
import numpy as np
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import Pair, to_gpu

pytestmark = pytest.mark.gpu

TOL = 1e-11   # asked of the solver, and so the bound on the oracle's residual (FP64 rounding is 1e-15)

FORMS = [(lqcd.F64, lqcd.F64, lqcd.F64), (lqcd.F32, lqcd.F32, lqcd.F64), (lqcd.F16S, lqcd.F32, lqcd.F64),
         (lqcd.F64, lqcd.F32, lqcd.F32), (lqcd.F32, lqcd.F32, lqcd.F32), (lqcd.F16S, lqcd.F32, lqcd.F32)]


@pytest.mark.parametrize("form", FORMS, ids=lambda f: "sap%d-inner%d-krylov%d" % f)
def test_even_gcr(form):
    sap_prec, inner, krylov = form
    P = Pair((8, 4, 12, 4), kappa=0.1355)
    eta = synth.gaussian_spinor(3 * P.Vh, 41).reshape(3, P.Vh, 4, 3)
    eta[1] = 0
    kw = dict(tol=TOL, sap_prec=sap_prec, inner=inner, krylov=krylov)
    psi, info, st = P.ctx.solve_dhat(to_gpu(eta), **kw)
    assert st == 0 and [i["status"] for i in info] == [0, 0, 0]
    assert torch.count_nonzero(psi[1]).item() == 0 and info[1]["iters"] == 0
    for k in (0, 2):
        r = np.linalg.norm(P.o.Dhat(psi[k].cpu().numpy()) - eta[k]) / np.linalg.norm(eta[k])
        assert r <= TOL * (1 + 1e-3)
        assert abs(info[k]["relres_dhat"] - r) <= 1e-3 * TOL
    x0 = psi * (1 + 1e-3)
    x0[1] = 0
    gsi, ginfo, st = P.ctx.solve_dhat_guess(to_gpu(eta), x0, **kw)
    assert st == 0
    for k in (0, 2):
        r = np.linalg.norm(P.o.Dhat(gsi[k].cpu().numpy()) - eta[k]) / np.linalg.norm(eta[k])
        assert r <= TOL * (1 + 1e-3)
        assert ginfo[k]["iters"] < info[k]["iters"]   # three digits are there already
