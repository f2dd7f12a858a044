"""CGNR where the recursive residual reaches the tolerance and the true one does not: the
solve starts again from the true residual until the iteration limit, wherever in a
group of four iterations the limit falls, and reports that it did not converge."""
import pytest

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import Pair, to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def pair():
    return Pair((4, 4, 4, 4))


@pytest.mark.parametrize("nmx", [40, 41, 42, 43, 200, 201, 202, 203])
def test_limit_after_restarts(pair, nmx):
    eta = to_gpu(synth.gaussian_spinor(pair.Vh, 63))
    _, info, st = pair.ctx.solve_dhat(eta, solver=lqcd.SOLVER_CGNR, tol=1e-16, nmx=nmx, check=False)
    assert st == 5 and info[0]["status"] == 5 and info[0]["iters"] == nmx
    # past its 120th iteration the true residual is within a few hundred roundings of zero
    assert nmx < 100 or info[0]["relres_dhat"] < 1e-13
