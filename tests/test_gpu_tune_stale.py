"""A cache file written when the kernels behind its keys were older ones (keys without the
generation of the kernels) decides nothing: the first call searches."""
import json

import pytest
import torch

from paper_1011_0911_gb300 import lqcd, synth
from tests.gpu_util import links, to_gpu

pytestmark = pytest.mark.gpu


def test_entries_of_older_kernels(tmp_path, monkeypatch, capfd):
    dims = (4, 4, 4, 6)
    gpu = torch.cuda.get_device_name().replace(" ", "_")
    shape = "x".join(map(str, dims))
    old = {f"k_hop4/m{m}/p1/n1/{shape}/{gpu}": [0, 32, 1, 0.1, 1, 0] for m in (1, 2)}
    cache = tmp_path / "tune.json"
    cache.write_text("{\n" + ",\n".join(f'  "{k}": {json.dumps(v)}' for k, v in old.items()) + "\n}\n")
    monkeypatch.setenv("LQCD_TUNE_CACHE", str(cache))
    monkeypatch.setenv("LQCD_TUNE_VERBOSE", "1")
    for v in ("LQCD_TUNE", "LQCD_HOP_KIND"):
        monkeypatch.delenv(v, raising=False)
    lqcd.tune_reset()
    ctx = lqcd.Context(dims)
    ctx.set_gauge(to_gpu(links(dims, 5)))
    ctx.clover_invert(0.1355, 1.9)
    x = to_gpu(synth.gaussian_spinor(ctx.Vh, 85), lqcd.F32)
    ctx.apply_Dhat(x, lqcd.F32)
    torch.cuda.synchronize()
    err = capfd.readouterr().err
    lqcd.tune_reset()
    for k in old:
        assert f"tune {k}" in err, k
    kept = json.loads(cache.read_text())
    assert len([k for k in kept if k.startswith("k_hop4/m1/p1/n1/")]) == 2
