"""The launch autotuner's search and cache, on the CPU: the timer is replaced by a model and the plan's
tuning calls are recorded, so nothing is launched."""
import json

import pytest

from paper_2101_10296_gb300 import autotune
from paper_2101_10296_gb300 import inputs as I

torch = pytest.importorskip("torch")


@pytest.fixture
def timed(qlib, monkeypatch):
    """(plan factory, {tuning: ms} model): autotune.autotune with the model's times."""
    model = {}

    class Recorder(qlib.Plan):
        def set_tuning(self, **t):
            self.tuning = t

    monkeypatch.setattr(autotune, "_time", lambda plan, params, grad, reps: model["ms"](plan.tuning))
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda *a: "test device")
    return Recorder, model


@pytest.mark.parametrize("graph,p,grad", [
    (I.random_regular(60, 3, 1), 1, True), (I.random_regular(60, 3, 1), 2, True), (I.random_regular(60, 3, 1), 2, False),
    (I.cycle(20), 3, True), (I.torus(6, 6), 3, True)],
    ids=["depth-1", "depth-2", "depth-2-energy", "general", "large-state"])
@pytest.mark.parametrize("P", [1, 33])
def test_the_default_is_a_candidate(timed, tmp_path, graph, p, grad, P):
    """Where no value is faster than the library's own choice (0), the search keeps it: autotuning does
    not leave a plan slower than not tuning it."""
    make, model = timed
    plan = make(graph, p)
    params = torch.zeros(1, P, 2 * p, dtype=torch.float64)
    model["ms"] = lambda t: 1.0 + 0.1 * (t["points_per_task"] != 0) + 0.1 * (t["blocks_per_sm"] != 0)
    best, results = autotune.autotune(plan, params, grad=grad, cache_path=str(tmp_path / "c.json"))
    assert best["points_per_task"] == 0 and best["blocks_per_sm"] == 0
    assert plan.tuning == best and results
    # and a faster value is still found, the largest too: the library cuts what does not fit
    model["ms"] = lambda t: 1.0 + abs(t["points_per_task"] - min(32, P)) + 0.1 * abs(t["blocks_per_sm"] - 2)
    best, _ = autotune.autotune(plan, params, grad=grad, cache_path=None, use_cache=False)
    assert best["points_per_task"] == min(32, P) and best["blocks_per_sm"] == 2


def test_the_cache_is_of_these_kernels(timed, tmp_path, monkeypatch):
    """A stored choice answers for the library that was timed, the plan's shape and its cut values' range
    (which sets the kernels' table rows): another library searches again."""
    make, model = timed
    cache = str(tmp_path / "c.json")
    plan = make(I.star(8), 1)
    params = torch.zeros(1, 16, 2, dtype=torch.float64)
    model["ms"] = lambda t: 1.0 + abs(t["points_per_task"] - 4)
    best, results = autotune.autotune(plan, params, cache_path=cache)
    assert best["points_per_task"] == 4 and results
    assert autotune.autotune(plan, params, cache_path=cache) == (best, {})
    wide = make(I.star(8), 1, weights=[[8] * 8])  # 64 cut bits instead of 8, else the same shape
    assert autotune.autotune(wide, params, cache_path=cache)[1]
    monkeypatch.setattr(autotune, "_kernels", lambda: "another library")
    model["ms"] = lambda t: 1.0 + abs(t["points_per_task"] - 8)
    best, results = autotune.autotune(plan, params, cache_path=cache)
    assert best["points_per_task"] == 8 and results
    assert len(json.load(open(cache))) == 3
