"""The walk's evaluation has one form, so that choosing parameters must not run
anything: tuned_params without a cache entry, with one, and with walk_eval given;
tune_walk times its form once, early and late in the run."""
import json

import pytest


@pytest.fixture
def autotune(tmp_path, monkeypatch):
    from paper_2005_05328_gb300 import autotune as a
    from paper_2005_05328_gb300 import build
    build.build()
    monkeypatch.setenv("DZS_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(a, "_gpu_name", lambda device: "GPU")
    a.timed = []
    monkeypatch.setattr(a, "_walk_ms", lambda p, warm, steps: a.timed.append((warm, steps)) or 1.5)
    yield a
    del a.timed


def test_tuned_params_runs_nothing(autotune):
    import paper_2005_05328_gb300 as dzs
    assert autotune.tuned_params(n1d=32, mesh=64, box=64.0).walk_eval == dzs.WALK_AUTO
    assert autotune.tuned_params(n1d=32, mesh=64, box=64.0, walk_eval=dzs.WALK_GUARDED).walk_eval == dzs.WALK_GUARDED
    assert autotune.timed == []


def test_tune_walk_times_once_and_is_used(autotune, tmp_path):
    import paper_2005_05328_gb300 as dzs
    mode = autotune.tune_walk(32, 64, 64.0, theta=0.4)
    assert mode in (dzs.WALK_MASKED, dzs.WALK_GUARDED)
    assert autotune.timed == [(2, 3), (76, 3)]  # 0.8 of the 96 steps
    (entry,) = json.load(open(tmp_path / "tune.json")).values()
    assert entry["walk_eval"] == mode and set(entry["ms"].values()) == {3.0}
    assert autotune.tune_walk(32, 64, 64.0, theta=0.4) == mode
    P = autotune.tuned_params(n1d=32, mesh=64, box=64.0, theta=0.4, seed=5)
    assert P.walk_eval == mode and P.theta == 0.4
    assert autotune.tuned_params(n1d=32, mesh=64, box=64.0).walk_eval == dzs.WALK_AUTO  # another shape
    assert len(autotune.timed) == 2
