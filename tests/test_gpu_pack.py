"""Canonical <-> native conversion: the tiled kernel against the documented
native layout and against the kernel for canonical fields off 16-byte
alignment; ranks that end in a partial tile, lattices smaller than one tile."""
import ctypes as C

import numpy as np
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests import util

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 4, 6), (6, 6, 6, 4), (10, 6, 4, 6), (8, 8, 8, 8)],
                         ids=lambda d: "x".join(map(str, d)))
@pytest.mark.parametrize("prec", [lqcd.F64, lqcd.F32, lqcd.F16S], ids=["f64", "f32", "f16s"])
def test_pack_layout_and_alignment(dims, prec):
    ctx = lqcd.Context(dims)
    ev, od = util.even_odd_sites(dims)
    n = 3
    dt = torch.complex128 if prec == lqcd.F64 else torch.complex64
    real = torch.float64 if prec == lqcd.F64 else torch.float32
    for nsub in (1, 2):
        ns = nsub * ctx.Vh
        x = torch.from_numpy(synth.gaussian_spinor(n * ns, 7).reshape(n, ns, 4, 3)).to(dt).cuda()
        nat = ctx.pack(x, prec, nsub)
        if prec != lqcd.F16S:   # word q of rank r of half h: [(h W + q) Vh + r]
            w = 1 if prec == lqcd.F64 else 2
            v = x.reshape(n, ns, 12)
            half = [v[:, ev], v[:, od]] if nsub == 2 else [v]
            ref = torch.stack([h.reshape(n, ctx.Vh, 12 // w, w).transpose(1, 2) for h in half], 1)
            assert torch.equal(nat.view(real), torch.view_as_real(ref.contiguous()).reshape(-1))
            assert torch.equal(ctx.unpack(nat, prec, nsub, n).reshape(x.shape), x)
        # the same bytes from, and to, a canonical field 4 (F64: 8) bytes off alignment
        f = torch.zeros(2 * x.numel() + 1, dtype=real, device="cuda")
        f[1:] = torch.view_as_real(x).reshape(-1)
        off = C.c_void_p(f.data_ptr() + f.element_size())
        nat2 = torch.zeros_like(nat)
        lib = lqcd.lib()
        assert lib.lqcd_pack(ctx._h, prec, nsub, off, C.c_void_p(nat2.data_ptr()), n) == 0
        assert torch.equal(nat2, nat)
        back = ctx.unpack(nat, prec, nsub, n)
        assert lib.lqcd_unpack(ctx._h, prec, nsub, C.c_void_p(nat.data_ptr()), off, n) == 0
        torch.cuda.synchronize()
        assert torch.equal(f[1:], torch.view_as_real(back).reshape(-1))
        assert float(f[0]) == 0.0 and np.isfinite(float(f.sum()))
