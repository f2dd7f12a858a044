"""Force kernels at the edges of their launch tiles: 64 or 128 ranks of one
parity per CTA, one row of CTAs per (direction, parity)."""
import numpy as np
import pytest

from paper_1011_0911_gb300 import synth
from tests import util
from tests.gpu_util import Pair, to_gpu

pytestmark = pytest.mark.gpu

# FP64 sums of a few hundred products of O(1) terms: the bound of test_gpu_md.py
TOL = 1e-12


def cpu(t):
    return t.detach().cpu().numpy()


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 4, 2, 2), (2, 2, 6, 8)], ids=lambda d: "x".join(map(str, d)))
def test_forces_every_link(dims):
    """Fewer ranks than one CTA (8, 48, 96 per parity) and extents of 2, where
    forward and backward neighbours coincide; the log det force of each parity
    takes the two forms that leave out the other parity's sites."""
    P = Pair(dims, kappa=0.1355, csw=1.9, seed=21)
    X, Y = synth.gaussian_spinor(P.V, 22), synth.gaussian_spinor(P.V, 23)
    assert util.relerr(cpu(P.ctx.force_dD(to_gpu(X), to_gpu(Y))), P.o.force_dD(X, Y)) < TOL
    for parity in (0, 1):
        assert util.relerr(cpu(P.ctx.force_logdet(parity)), P.o.grad_logdet(parity)) < TOL
    assert util.relerr(cpu(P.ctx.force_gauge(5.3)), P.o.grad_gauge(5.3)) < TOL


def test_force_dD_ragged_sampled():
    """720 ranks per parity: several CTAs of each kernel and a partial last one."""
    P = Pair((6, 10, 6, 4), kappa=0.1355, csw=1.9, seed=24)
    X, Y = synth.gaussian_spinor(P.V, 25), synth.gaussian_spinor(P.V, 26)
    g = cpu(P.ctx.force_dD(to_gpu(X), to_gpu(Y)))
    rng = np.random.default_rng(5)
    samples = [(P.V - 1, m, 7 - m) for m in range(4)] + [(P.V - 2, m, m) for m in range(4)]
    samples += [(int(rng.integers(P.V)), int(rng.integers(4)), int(rng.integers(8))) for _ in range(16)]
    for x, mu, a in samples:
        ref = np.vdot(Y, P.o.dD_apply(X, x, mu, a)).real
        assert abs(g[x, mu, a] - ref) <= TOL * max(1.0, abs(ref)), (x, mu, a)
