"""The FP64 stencil's splits of a site over 2, 4 and 8 threads: each against the
oracle, and all bitwise equal (they add in one order), on lattices whose ranks
fill less than one warp, end in a partial warp, or wrap in two hops."""
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import TOL, Pair, relerr, to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 4, 2), (6, 6, 6, 4), (10, 6, 4, 6)],
                         ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("nrhs", [1, 3])
def test_splits(dims, nrhs, monkeypatch):
    P = Pair(dims)
    x = synth.gaussian_spinor(nrhs * P.V, 31).reshape(nrhs, P.V, 4, 3)
    e = synth.gaussian_spinor(nrhs * P.Vh, 32).reshape(nrhs, P.Vh, 4, 3)
    first = None
    for split in ("d1", "d2", "d4"):
        monkeypatch.setenv("LQCD_HOP_KIND", split)
        d, dh = P.ctx.apply_D(to_gpu(x)), P.ctx.apply_Dhat(to_gpu(e))
        w = P.ctx.apply_W(to_gpu(e), 0.1)
        if first is None:
            first = (d, dh, w)
            for k in range(nrhs):
                assert relerr(d[k], P.o.D(x[k])) < TOL[lqcd.F64]
                assert relerr(dh[k], P.o.Dhat(e[k])) < TOL[lqcd.F64]
        for a, b in zip(first, (d, dh, w)):
            assert torch.equal(a, b), split
