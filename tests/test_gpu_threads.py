"""Two host threads, each with a context on a stream of its own, at kernels that both use
with different amounts of shared memory: every call gives the bits of the same call
made alone."""
import threading

import numpy as np
import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import links, to_gpu

pytestmark = pytest.mark.gpu

DIMS = (8, 4, 4, 4)


def context(stream):
    ctx = lqcd.Context(DIMS, stream=stream)
    with torch.cuda.stream(stream):
        ctx.set_gauge(to_gpu(links(DIMS, 5)))
        ctx.clover_invert(0.1355, 1.9)
    return ctx


def together(calls, reps):
    """calls: (stream, function) pairs; every function's results reps times over, the threads at once."""
    start, out, errors = threading.Barrier(len(calls)), [None] * len(calls), []

    def work(i):
        stream, fn = calls[i]
        try:
            with torch.cuda.stream(stream):
                start.wait()
                out[i] = [fn() for _ in range(reps)]
                stream.synchronize()
        except Exception as e:   # noqa: BLE001 - reported by the test
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    return out


@pytest.mark.parametrize("act", [lqcd.F32, lqcd.BF16], ids=["f32", "bf16"])
def test_network_layers(act):
    calls = []
    for i, chans in enumerate([(1, 1), (1, 2, 2, 1)]):
        stream = torch.cuda.Stream()
        ctx = context(stream)
        rng = np.random.default_rng(i)
        n = ctx.net_weight_count(chans)
        ctx.net_set(chans, (0.1 * (rng.standard_normal(n) + 1j * rng.standard_normal(n))).astype(np.complex64), act=act)
        x = to_gpu(synth.gaussian_spinor(ctx.V, 70 + i))
        torch.cuda.synchronize()
        calls.append((stream, lambda ctx=ctx, x=x: ctx.net_apply(x)))
    alone = [together([c], 1)[0][0] for c in calls]
    for ref, out in zip(alone, together(calls, 400)):
        assert all(torch.equal(ref, y) for y in out)


def test_little_operator_build():
    calls = []
    for i, (bs, ns) in enumerate([((4, 4, 4, 4), 24), ((2, 4, 2, 2), 4)]):
        stream = torch.cuda.Stream()
        ctx = context(stream)
        v0 = to_gpu(synth.gaussian_spinor(ns * ctx.V, 80 + i).reshape(ns, ctx.V, 4, 3))
        torch.cuda.synchronize()

        def build(ctx=ctx, bs=bs, v0=v0):
            ctx.dfl_build(v0, bs=bs, ninv=1, ncy=1, nmr=2, prec=lqcd.F32, coarse_prec=lqcd.F32, coarse_tol=1e-5)
            return ctx.dfl_export()[1]
        calls.append((stream, build))
    alone = [together([c], 1)[0][0] for c in calls]
    for ref, out in zip(alone, together(calls, 30)):
        assert all(torch.equal(ref, y) for y in out)
