"""The autotuner's file of winners: used again for the same size class and the
same kernels, not for an entry that other kernels were timed for."""
import json

import torch

from paper_2609_40159_gb300 import autotune
from test_autotune_host import _FakePlan

MODES, RPWS, KTS = ("level", "hybrid"), (4, 32), (1,)


def _tune(monkeypatch, times):
    plan = _FakePlan(times)
    monkeypatch.setattr(autotune, "time_call", lambda fn, reps=5: times[plan.choice])
    res = autotune.tune_plan(plan, torch.zeros(10_000, 1, dtype=torch.float64), modes=MODES, rpws=RPWS, kts=KTS)
    return res, plan


def test_cache_is_bound_to_the_kernels(monkeypatch, tmp_path):
    path = tmp_path / "tune.json"
    monkeypatch.setenv("SPTRSV_TUNE_CACHE", str(path))
    times = {(m, r, 1): 2.0 for m in MODES for r in RPWS}
    times[("level", 32, 1)] = 1.0
    # an entry as it was written before the kernels were part of the key
    key = autotune.size_class(10_000, 50_000, 100, 1, torch.float64)
    path.write_text(json.dumps({key: dict(mode="hybrid", rows_per_warp=4, rhs_tile=1, ms=0.1)}))
    res, plan = _tune(monkeypatch, times)
    assert not res["cached"] and plan.choice == ("level", 32, 1)
    res, plan = _tune(monkeypatch, dict.fromkeys(times, 9.0))
    assert res["cached"] and plan.choice == ("level", 32, 1) and res["key"] == key
    # other kernels: timed again, the first ones' winner is kept beside
    monkeypatch.setattr(autotune, "kernel_version", lambda: "other")
    times[("hybrid", 32, 1)] = 0.5
    res, plan = _tune(monkeypatch, times)
    assert not res["cached"] and plan.choice == ("hybrid", 32, 1)
    monkeypatch.undo()
    monkeypatch.setenv("SPTRSV_TUNE_CACHE", str(path))
    res, plan = _tune(monkeypatch, times)
    assert res["cached"] and plan.choice == ("level", 32, 1)


def test_kernel_version_follows_the_sources():
    v = autotune.kernel_version()
    assert len(v) == 12 and v == autotune.kernel_version()
