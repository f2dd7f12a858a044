"""CGNR with its scalars on the device: the iterate and the count at any iteration
limit are those of a plain CG in FP64 (numpy, the oracle's Dhat), although the
host runs ahead; zero and non-finite sources; lattices of a few CTAs."""
import numpy as np
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests import util
from tests.gpu_util import Pair, to_gpu

pytestmark = pytest.mark.gpu

G5 = np.array([1, 1, -1, -1.0])[:, None]


def cg(P, eta, n):
    x, r = np.zeros_like(eta), eta.copy()
    dag = lambda v: G5 * P.o.Dhat(G5 * v)   # noqa: E731
    z = dag(r)
    p, zz = z.copy(), np.vdot(z, z).real
    for _ in range(n):
        w = P.o.Dhat(p)
        a = zz / np.vdot(w, w).real
        x, r = x + a * p, r - a * w
        z = dag(r)
        z2 = np.vdot(z, z).real
        p, zz = z + (z2 / zz) * p, z2
    return x


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 6, 6, 4)], ids=lambda d: "x".join(map(str, d)))
def test_iterates(dims):
    P = Pair(dims, kappa=0.13)
    eta = synth.gaussian_spinor(P.Vh, 61)
    for n in (0, 1, 2, 3, 7):
        psi, info, st = P.ctx.solve_dhat(to_gpu(eta), solver=lqcd.SOLVER_CGNR, tol=1e-14, nmx=n, check=False)
        assert st == 5 and info[0]["iters"] == n
        ref = cg(P, eta, n)
        if n == 0:
            assert torch.count_nonzero(psi).item() == 0
        else:   # a few steps of rounding at 1e-16 each
            assert util.relerr(psi.cpu().numpy(), ref) < 1e-13
        assert abs(info[0]["relres_dhat"] - np.linalg.norm(eta - P.o.Dhat(ref)) / np.linalg.norm(eta)) < 1e-12
    psi, info, st = P.ctx.solve_dhat(to_gpu(eta), solver=lqcd.SOLVER_CGNR, tol=1e-12, nmx=1000)
    assert st == 0 and info[0]["relres_dhat"] <= 1e-12
    assert util.relerr(P.o.Dhat(psi.cpu().numpy()), eta) <= 1.01e-12


def test_sources_without_a_solution():
    P = Pair((2, 2, 2, 2))
    eta = synth.gaussian_spinor(2 * P.Vh, 62).reshape(2, P.Vh, 4, 3)
    eta[0] = 0
    psi, info, st = P.ctx.solve_dhat(to_gpu(eta), solver=lqcd.SOLVER_CGNR, tol=1e-10, nmx=1000)
    assert st == 0 and info[0]["iters"] == 0 and info[1]["iters"] > 0
    assert torch.count_nonzero(psi[0]).item() == 0
    eta[1, 3, 2, 1] = np.nan
    _, info, st = P.ctx.solve_dhat(to_gpu(eta), solver=lqcd.SOLVER_CGNR, tol=1e-10, nmx=1000, check=False)
    assert st == 7 and info[0]["status"] == 0 and info[1]["status"] == 7
