"""A source that is not finite: its lattice is reported as such (status 7, as by the
single-lattice solver), the other lattices of the batch are solved."""
import numpy as np
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests import util
from tests.gpu_util import Pair, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bad", [np.nan, np.inf, 1e200], ids=["nan", "inf", "overflow"])
def test_one_source_not_finite(bad):
    pairs = [Pair((8, 8, 8, 8), kappa=0.1350, seed=1), Pair((12, 8, 8, 8), kappa=0.1355, seed=3)]
    eta = [synth.gaussian_spinor(P.Vh, 750 + i).reshape(P.Vh, 4, 3) for i, P in enumerate(pairs)]
    eta[0][5, 2, 1] = bad
    _, one, st1 = pairs[0].ctx.solve_dhat(to_gpu(eta[0]), sap_prec=lqcd.F32, inner=lqcd.F32, check=False)
    assert st1 == 7 and one[0]["status"] == 7
    B = lqcd.Batch([P.ctx for P in pairs])
    psi, info, st = B.solve_dhat([to_gpu(e) for e in eta])
    assert st == 7 and [i["status"] for i in info] == [7, 0]
    assert info[0]["iters"] == 0 and torch.count_nonzero(psi[0]).item() == 0
    assert info[1]["relres_dhat"] <= 1e-10
    assert util.relerr(pairs[1].o.Dhat(psi[1].cpu().numpy()), eta[1]) <= 1e-10
