"""FP16 fields whose sites are as small as floats get: a site is held to the rounding of a
half (2^-11 of its largest component, and 2^-149, the spacing of the smallest floats)
above 2^-128, where the inverse of its scale leaves float's range, and is zero below."""
import numpy as np
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import to_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("aligned", [True, False], ids=["tiled", "plain"])
def test_round_trip(aligned):
    dims = (4, 4, 4, 6)
    V = dims[0] * dims[1] * dims[2] * dims[3]
    ctx = lqcd.Context(dims)
    x = synth.gaussian_spinor(V, 83).reshape(V, 12)
    x /= np.maximum(abs(x.real), abs(x.imag)).max(1, keepdims=True)   # the largest component is 1
    top = np.ldexp(1 + (np.arange(V) % 7) / 7, -120 - np.arange(V) % 28)   # 2^-120 .. 2^-147
    x = (x * top[:, None]).astype(np.complex64)
    t = to_gpu(x, lqcd.F32).reshape(1, V, 4, 3)
    if not aligned:   # a canonical field on an 8-byte boundary takes another conversion kernel
        b = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)[1:].view(t.shape)
        t = b.copy_(t)
        assert t.data_ptr() % 16 == 8
    out = ctx.unpack(ctx.pack(t, lqcd.F16S, 2), lqcd.F16S, 2, 1).cpu().numpy().reshape(V, 12)
    m = np.maximum(abs(x.real), abs(x.imag)).max(1).astype(np.float64)
    held = m > 2.0 ** -128
    assert held.any() and not held.all()
    bound = (2.0 ** -11 + 2.0 ** -22) * m[held] + 2.0 ** -149
    err = np.maximum(abs(out.real.astype(np.float64) - x.real), abs(out.imag.astype(np.float64) - x.imag)).max(1)
    assert (err[held] <= bound).all()
    assert np.count_nonzero(out[~held]) == 0
