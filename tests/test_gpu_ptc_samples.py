"""The BF16 layers keep a tile of sites for several samples: with many samples in
a call every sample's result is that of a call of its own, bit for bit, on
lattices whose last tile is partial and for one and two channels."""
import numpy as np
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import Pair
from tests.test_gpu_ptc import rand_weights

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chans", [(1, 1), (1, 2, 1), (1, 2, 2, 1)], ids=str)
@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (6, 6, 6, 6), (16, 8, 8, 12)], ids=lambda d: "x".join(map(str, d)))
def test_samples(dims, chans):
    P = Pair(dims)
    P.ctx.net_set(chans, rand_weights(chans, 5, ident=0.8), act=lqcd.BF16)
    n = 23 if P.V > 10000 else 5   # 192 tiles x 23 samples: two samples per CTA, one left over
    x = torch.from_numpy(np.stack([synth.gaussian_spinor(P.V, 80 + k) for k in range(n)])).cuda()
    many = P.ctx.net_apply(x)
    for k in range(n):
        assert torch.equal(P.ctx.net_apply(x[k:k + 1]).reshape(-1), many[k].reshape(-1)), k
