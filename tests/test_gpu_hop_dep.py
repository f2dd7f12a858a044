"""D and Dhat with their kernels launched dependently or plainly: the same bits; without a
recorded choice both are timed, the faster one is kept (dependent launches where they
are at most 5 % slower), persists in the cache file and is read back."""
import json
import re

import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import links, to_gpu

pytestmark = pytest.mark.gpu

DIMS = (16, 8, 8, 8)
NRHS = 3
LINE = re.compile(r"tune (\S+): dependent=(\d) ([0-9.]+) us")


@pytest.mark.parametrize("prec", [lqcd.F64, lqcd.F32, lqcd.F16S], ids=["f64", "f32", "f16s"])
@pytest.mark.parametrize("op", ["Dhat", "D"])
def test_choice(op, prec, tmp_path, monkeypatch, capfd):
    cache = tmp_path / "tune.json"
    monkeypatch.setenv("LQCD_TUNE_CACHE", str(cache))
    monkeypatch.setenv("LQCD_TUNE_VERBOSE", "1")
    for v in ("LQCD_TUNE", "LQCD_HOP_KIND"):
        monkeypatch.delenv(v, raising=False)
    lqcd.tune_reset()
    ctx = lqcd.Context(DIMS)
    ctx.set_gauge(to_gpu(links(DIMS, 5)))
    ctx.clover_invert(0.1355, 1.9)
    x = to_gpu(synth.gaussian_spinor(NRHS * (ctx.Vh if op == "Dhat" else ctx.V), 86), prec).reshape(NRHS, -1, 4, 3)
    apply = (lambda: ctx.apply_Dhat(x, prec)) if op == "Dhat" else (lambda: ctx.apply_D(x, prec))
    first = apply()
    torch.cuda.synchronize()
    head = f"k_hop_dep/m{0 if op == 'Dhat' else 1}/p{prec}/n{NRHS}/"
    times = {"0": [], "1": []}
    for line in capfd.readouterr().err.splitlines():
        m = LINE.match(line)
        if m and m[1].startswith(head):
            times[m[2]].append(float(m[3]))
    assert len(times["0"]) == len(times["1"]) == 2
    entries = json.loads(cache.read_text())
    (key,) = [k for k in entries if k.startswith(head)]
    plain, dep = min(times["0"]), min(times["1"])
    # printed to 0.1 us
    assert dep <= 1.05 * plain + 0.11 if entries[key][0] else dep >= 1.05 * plain - 0.11
    for choice in (0, 1):
        entries[key][0] = choice
        cache.write_text("{\n" + ",\n".join(f'  "{k}": {json.dumps(v)}' for k, v in entries.items()) + "\n}\n")
        lqcd.tune_reset()
        again = apply()
        torch.cuda.synchronize()
        assert torch.equal(again, first)
        assert f"tune {head}" not in capfd.readouterr().err
    lqcd.tune_reset()
