"""The plan cache on a CPU: a plan is kept for the version of the library that measured it."""
import json
from types import SimpleNamespace

import pytest


@pytest.fixture
def cache(monkeypatch):
    import paper_1403_0734_gb300.build as kb
    kb.build()
    from paper_1403_0734_gb300 import kc
    calls = SimpleNamespace(tuned=0, applied=[])

    def tune(g, k, per_vertex=False, stream=None):
        calls.tuned += 1
        return {"k": k, "per_vertex": per_vertex, "algo": [1] * 7, "parts": [calls.tuned] * 7, "ms": [0.0] * 7}

    monkeypatch.setattr(kc, "tune", tune)
    monkeypatch.setattr(kc, "set_tuning", lambda g, p: calls.applied.append(p))
    return kc, calls


G = SimpleNamespace(n=10, m=20, max_dplus=5, wedges=30)


def test_plan_is_measured_once_and_kept(cache, tmp_path):
    kc, calls = cache
    path = str(tmp_path / "plans.json")
    p = kc.TuningCache(path).plan(G, 5)
    assert kc.TuningCache(path).plan(G, 5) == p and calls.tuned == 1
    assert kc.TuningCache(path).plan(G, 5, per_vertex=True) != p and calls.tuned == 2
    assert [a["parts"][0] for a in calls.applied] == [1, 1, 2]


@pytest.mark.parametrize("lib", [None, "kc 0.1 sm_103a"])
def test_plan_of_another_version_is_measured_again(cache, tmp_path, lib):
    kc, calls = cache
    path = str(tmp_path / "plans.json")
    old = {"k": 5, "per_vertex": False, "algo": [0] * 7, "parts": [9] * 7, "ms": [1.0] * 7}
    if lib:
        old["lib"] = lib
    with open(path, "w") as f:
        json.dump({kc.TuningCache.key(G, 5, False): old, "other": old}, f)
    p = kc.TuningCache(path).plan(G, 5)
    assert calls.tuned == 1 and p["parts"] == [1] * 7 and calls.applied == [p]
    with open(path) as f:
        kept = json.load(f)
    assert kept["other"] == old and kept[kc.TuningCache.key(G, 5, False)] == p
    assert kc.TuningCache(path).plan(G, 5) == p and calls.tuned == 1
