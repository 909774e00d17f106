"""The autotuner's cache key tells apart whatever takes another instantiation of the TMA kernel, and plans
that were timed before its costs changed are not taken."""
import json

import pytest

from paper_2201_06039_gb300 import lbm


def _lattice(monkeypatch, **kw):
    import torch
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda d: "Some GPU")
    lat = lbm.Lattice.__new__(lbm.Lattice)
    lat.params = lbm.lbm_params_default()
    lat.params.nx, lat.params.ny, lat.params.nz = 32, 32, 32
    for k, v in kw.items():
        setattr(lat.params, k, v)
    return lat


@pytest.mark.parametrize("kw", [dict(thermal_off=1), dict(precision=1), dict(nz=33), dict(wall_scheme=1)])
def test_plan_key_tells_instantiations_apart(monkeypatch, kw):
    assert _lattice(monkeypatch, **kw).plan_key() != _lattice(monkeypatch).plan_key()


def test_a_plan_of_an_earlier_kernel_is_timed_again(monkeypatch, tmp_path):
    cache = tmp_path / "plans.json"
    old = "32x32x32/prec0/bc000000/wet0/Some_GPU"     # key and plan of 16-plane chunks, as they were written
    cache.write_text(json.dumps({old: dict(shape=0, zchunk=16, ms_per_step=0.045, steps=10)}))
    lat = _lattice(monkeypatch)
    lat.ctx = None
    monkeypatch.setattr(lbm, "lbm_autotune", lambda ctx, steps: 0.012)
    monkeypatch.setattr(lbm, "lbm_get_plan", lambda ctx: (0, 1, 128, 128))
    monkeypatch.setattr(lbm, "lbm_select_plan", lambda *a: pytest.fail("took a plan of another kernel"))
    res = lat.autotune(steps=5, cache=str(cache))
    assert res == dict(shape=0, zchunk=1, ms_per_step=0.012, cached=False)
    table = json.loads(cache.read_text())
    assert table[old]["zchunk"] == 16 and table[lat.plan_key()]["zchunk"] == 1
    taken = []
    monkeypatch.setattr(lbm, "lbm_select_plan", lambda ctx, *plan: taken.append(plan))
    assert lat.autotune(cache=str(cache))["cached"] and taken == [(0, 1)]
