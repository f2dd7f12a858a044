"""FP64 block solves with four threads a site against the one-thread-a-site kernel:
block shapes from 8 to 128 sites of a parity (partly filled warps, blocks that span
a direction, 2 sites deep), no, one and several steps, a source that is zero on most
blocks.  Both are FP64 orderings of the same sums: some thousand roundings of 1e-16
through a well-conditioned block operator, so 1e-12."""
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import links, to_gpu, util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,bs", [((8, 8, 8, 8), (4, 4, 4, 4)), ((8, 4, 12, 4), (2, 4, 6, 4)),
                                     ((8, 4, 12, 4), (4, 4, 6, 2)), ((4, 8, 4, 8), (2, 2, 2, 2)),
                                     ((4, 4, 4, 4), (4, 4, 4, 4)), ((12, 6, 4, 4), (6, 2, 2, 4)),
                                     ((8, 8, 2, 16), (2, 4, 2, 8))],
                         ids=lambda v: "x".join(map(str, v)))
@pytest.mark.parametrize("periodic", [False, True], ids=["antiperiodic", "periodic"])
def test_matches_the_general_kernel(dims, bs, periodic, monkeypatch):
    V = dims[0] * dims[1] * dims[2] * dims[3]
    ctx = lqcd.Context(dims, antiperiodic_t=not periodic)
    ctx.set_gauge(to_gpu(links(dims, 3)))
    ctx.clover_invert(0.1355, 1.9)
    eta = to_gpu(synth.gaussian_spinor(V, 61))
    one = torch.zeros_like(eta)
    one.view(-1)[:12] = eta.view(-1)[:12]
    for src, ncy, nmr in ((eta, 3, 5), (eta, 1, 0), (eta, 2, 1), (one, 2, 4)):
        out = []
        for generic in ("0", "1"):
            monkeypatch.setenv("LQCD_SAP_GENERIC", generic)
            out.append(ctx.sap(src, bs=bs, ncy=ncy, nmr=nmr, prec=lqcd.F64).cpu().numpy())
        assert util.relerr(out[0], out[1]) < 1e-12, (ncy, nmr)
