"""A cached launch is for handles that can take it: the options that select
other kernels, and the build that was timed, are part of the key, and a choice
the handle refuses is searched anew."""
import json

import pytest

from paper_1412_6238_gb300 import autotune
from paper_1412_6238_gb300 import workloads as wl


def test_keys():
    shapes = [(256, 128), (512, 256)]
    plain = autotune.cache_key("GB300", "f32", shapes)
    assert autotune.cache_key("GB300", "f32", shapes, ["", ""]) == plain
    keys = {autotune.cache_key("GB300", "f32", shapes, o, b)
            for o in (["", ""], ["d", ""], ["", "d"], ["v", "v"], ["rd", ""]) for b in ("", "x", "y")}
    assert len(keys) == 15


def drop(**options):
    w = wl.droplet(130, 60, 12.0, 65.0, 30.0, Re=0.2, Ma=10.0, Ca=0.05, eta_m=0.2, eta_r=0.5,
                   lam_r=0.5)
    w.params.update(options)
    return w


@pytest.mark.gpu
def test_options_and_refusals(tmp_path, monkeypatch):
    from paper_1412_6238_gb300.lbe import LBE
    path = tmp_path / "cache.json"
    monkeypatch.setenv("LBE_AUTOTUNE_CACHE", str(path))
    plain = autotune.tune(LBE(drop(), storage="f32"), steps=2, warmup=1)
    assert not plain["cached"]
    sim = LBE(drop(dissip=1), storage="f32")
    assert sim.options == ["d"]
    best = autotune.tune(sim, steps=2, warmup=1)
    assert not best["cached"] and best["kernel"] < 5  # (a strip kernel has no such term)
    assert autotune.tune(LBE(drop(dissip=1), storage="f32"), steps=2)["cached"]
    # every cached choice made one that no such handle takes
    cache = json.loads(path.read_text())
    assert len(cache) == 2
    path.write_text(json.dumps({k: dict(v, kernel=8, grid=0, seg_rows=0)
                                for k, v in cache.items()}))
    again = autotune.tune(LBE(drop(dissip=1), storage="f32"), steps=2, warmup=1)
    assert not again["cached"] and again["kernel"] < 5
