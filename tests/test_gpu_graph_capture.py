"""Calls recorded in a caller's CUDA graph: replayed after the links and the clover term
have changed they use the new operator, as an eager call does, and a call that is only
recorded leaves eager calls as they were."""
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import links, to_gpu

pytestmark = pytest.mark.gpu

DIMS = (8, 4, 4, 4)

CALLS = {
    "sap_f32": lambda c, x: c.sap(x, ncy=2, nmr=3, prec=lqcd.F32),
    "sap_f16s": lambda c, x: c.sap(x, ncy=2, nmr=3, prec=lqcd.F16S),
    "sap_f64": lambda c, x: c.sap(x, ncy=2, nmr=3, prec=lqcd.F64),
    "D_f64": lambda c, x: c.apply_D(x, lqcd.F64),
    "D_f32": lambda c, x: c.apply_D(x, lqcd.F32),
    "Dhat_f64": lambda c, x: c.apply_Dhat(x[: c.Vh], lqcd.F64),
    "Dhat_f16s": lambda c, x: c.apply_Dhat(x[: c.Vh], lqcd.F16S),
}


def set_operator(ctx, seed, kappa):
    ctx.set_gauge(to_gpu(links(DIMS, seed)))
    ctx.clover_invert(kappa, 1.9)


def recorded(ctx, fn, x, stream):
    fn(ctx, x)   # workspaces and launch shapes
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        out = fn(ctx, x)
    return graph, out


@pytest.mark.parametrize("name", CALLS)
def test_replay_follows_the_operator(name):
    fn = CALLS[name]
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx, ref = lqcd.Context(DIMS, stream=stream), lqcd.Context(DIMS, stream=stream)
        x = to_gpu(synth.gaussian_spinor(ctx.V, 84))
        if name in ("D_f32", "Dhat_f16s"):
            x = x.to(torch.complex64)
        set_operator(ctx, 5, 0.1355)
        first = fn(ctx, x).clone()
        graph, out = recorded(ctx, fn, x, stream)
        graph.replay()
        assert torch.equal(out, first)
        set_operator(ctx, 6, 0.1300)
        set_operator(ref, 6, 0.1300)
        graph.replay()
        want = fn(ref, x)
        assert torch.equal(out, want)
        assert not torch.equal(out, first)
        # changed again, recorded and not replayed: the eager call sees the operator of now
        set_operator(ctx, 7, 0.1320)
        set_operator(ref, 7, 0.1320)
        torch.cuda.synchronize()
        with torch.cuda.graph(torch.cuda.CUDAGraph(), stream=stream):
            fn(ctx, x)
        assert torch.equal(fn(ctx, x), fn(ref, x))
        torch.cuda.synchronize()
