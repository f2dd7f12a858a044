"""Clover inversion beyond the diagonal path: with a large c_sw some 6x6 blocks
need row exchanges; A, A^-1 and log det against the oracle's LU."""
import numpy as np
import pytest

from paper_1011_0911_gb300 import synth
from tests.gpu_util import Pair, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("csw", [0.0, 1.9, 9.0, 60.0])
def test_clover_inverse(csw):
    P = Pair((4, 2, 4, 6), kappa=0.1355, csw=csw, seed=31)
    pivots = 0
    for parity, sites in ((0, P.ev), (1, P.od)):
        x = synth.gaussian_spinor(P.Vh, 71 + parity)
        cond = 1.0
        for inverse in (False, True):
            got = P.ctx.apply_clover(parity, inverse, to_gpu(x)).cpu().numpy()
            for i, s in enumerate(sites):
                m = P.o.clover_site(s, inverse)
                ref = m @ x[i].ravel()
                if not inverse:
                    cond = max(cond, np.linalg.cond(m))
                    for b in (m[:6, :6], m[6:, 6:]):
                        pivots += np.abs(b[1:, 0]).max() > abs(b[0, 0])
                # LU in FP64: a few tens of roundings, amplified by the condition
                assert np.linalg.norm(got[i].ravel() - ref) <= 1e-14 * cond * np.linalg.norm(ref)
        assert abs(P.logdet[parity] - P.o.logdet(parity)) <= 1e-12 * max(1.0, abs(P.o.logdet(parity)))
    assert (pivots > 0) == (csw > 5)
