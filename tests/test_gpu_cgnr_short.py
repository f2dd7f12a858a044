"""CGNR solves of a few iterations: at most one iteration is launched beyond the one that
reaches the tolerance (a solve whose iteration limit is that very iteration can launch
none), whether the lattice is one that replays graphs or not."""
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import links, to_gpu

pytestmark = pytest.mark.gpu

PER_ITERATION = 8   # kernels


@pytest.mark.parametrize("dims", [(4, 4, 4, 4), (16, 8, 8, 8), (16, 16, 16, 12)], ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("tol", [0.7, 0.3, 0.1])
def test_launches(dims, tol):
    ctx = lqcd.Context(dims)
    ctx.set_gauge(to_gpu(links(dims, 5)))
    ctx.clover_invert(0.1355, 1.9)
    eta = to_gpu(synth.gaussian_spinor(ctx.Vh, 64))

    def solve(nmx):
        before = ctx.kernel_launches
        psi, info, st = ctx.solve_dhat(eta, solver=lqcd.SOLVER_CGNR, tol=tol, nmx=nmx)
        assert st == 0
        return psi, info[0]["iters"], ctx.kernel_launches - before

    solve(1000)   # launch shapes
    psi, iters, launches = solve(1000)
    ref, iters_ref, fewest = solve(iters)
    assert iters == iters_ref and 0 < iters < 10
    assert torch.equal(psi, ref)
    assert launches <= fewest + PER_ITERATION
