"""The autotuner and the library's one-launch path of small problems: host logic with faked
times, and on the GPU the choice it makes for a small problem."""
import json

import numpy as np
import pytest

from paper_1402_4089_gb300 import hmc, tune


def _fake(monkeypatch, tmp_path, own, tiled):
    import torch
    steps = []
    monkeypatch.setenv("HMC_TUNE_CACHE", str(tmp_path / "tune.json"))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "FakeGPU")
    monkeypatch.setattr(tune, "time_tile", lambda *a, **k: (
        (9.0, {"problems": [{}]}) if (a[8], a[9][0], a[9][3]) == (1, 4, 3) else (None, None)))

    def time_steps(*a, **k):
        steps.append((a[8], a[9]))
        return own if a[9] is None else tiled
    monkeypatch.setattr(tune, "time_steps", time_steps)
    return steps


@pytest.mark.parametrize("own,tiled,want", [(2.5, 10.0, (0, None)), (12.0, 10.0, (1, (4, 0, 0, 3))),
                                            (None, 10.0, (1, (4, 0, 0, 3)))])
def test_library_choice_is_compared_by_steps(monkeypatch, tmp_path, own, tiled, want):
    steps = _fake(monkeypatch, tmp_path, own, tiled)
    X, y = np.zeros((100, 10), np.float32), np.zeros(100, np.int32)
    assert tune.autotune(X, y, 2)[:2] == want
    assert steps == [(0, None)] + ([(1, (4, 0, 0, 3))] if own is not None else [])
    entry, = json.load(open(tmp_path / "tune.json")).values()
    assert entry["engine"] == want[0] and entry["tile"] == (list(want[1]) if want[1] else None)
    assert tune.autotune(X, y, 2)[:2] == want and len(steps) <= 2      # from the cache


def test_explicit_engine_and_reduced_precision_are_not_compared(monkeypatch, tmp_path):
    steps = _fake(monkeypatch, tmp_path, 1.0, 10.0)
    X, y = np.zeros((100, 10), np.float32), np.zeros(100, np.int32)
    assert tune.autotune(X, y, 2, engine=1)[:2] == (1, (4, 0, 0, 3))
    assert tune.autotune(X, y, 2, x_storage="bf16")[:2] == (1, (4, 0, 0, 3))
    assert steps == []


@pytest.mark.gpu
@pytest.mark.parametrize("n,p,K,xs,small", [(100, 10, 2, "f32", True), (1000, 50, 3, "f64", True),
                                            (20000, 300, 3, "f32", False)])
def test_small_problem_keeps_the_one_launch_path(cuda, n, p, K, xs, small):
    rng = np.random.default_rng(1)
    X = rng.standard_normal((n, p)).astype(np.float64 if xs == "f64" else np.float32)
    y = rng.integers(0, K, n).astype(np.int32)
    engine, tile, _ = tune.autotune(X, y, K, x_storage=xs, state=xs, reps=3, use_cache=False)
    assert (engine, tile) == (0, None) if small else tile is not None
    with hmc.create(X, y, K, x_storage=xs, state=xs, engine=engine, tile=tile) as h:
        assert bool(h.describe()["problems"][0].get("one_launch")) is small
