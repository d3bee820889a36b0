"""The tuner's probe and cache, with plans that only record what they are made of: each probe
has the form the tuned batch runs in (several branches), the library's own tiling (ctas = 0) is
among the candidates, and a cached table of another library is not used."""
import json

import pytest

from paper_2510_02635_gb300 import autotune
from paper_2510_02635_gb300 import workloads as W

torch = pytest.importorskip("torch")


@pytest.fixture
def probes(monkeypatch):
    made = []

    class Plan:
        def __init__(self, instances, branches=0, device="cuda"):
            self.ctas = instances[0]["problem"].ctas
            made.append((len(instances), branches, self.ctas))

        def close(self):
            pass

    monkeypatch.setattr(autotune.fbsde, "Plan", Plan)
    zeros = torch.zeros
    monkeypatch.setattr(torch, "zeros", lambda *a, **kw: zeros(*a, **{**kw, "device": "cpu"}))
    monkeypatch.setattr(autotune, "_library_hash", lambda: "here", raising=False)
    return made


def _instances():
    return [W.Workload("t", "ac_manufactured", d=300, sigma=1.0, T=0.5, N=4, M=16384, Q=1, seed=1,
                       x0_law="zero")]


def _times(monkeypatch, ms):
    monkeypatch.setattr(autotune, "_time_plan", lambda plan, torch, repeats: ms[plan.ctas])


def test_probe_has_the_form_of_the_batch(probes, monkeypatch):
    ms = {0: 1.0, 76: 2.0, 152: 1.5, 304: 1.3, 608: 1.02, 1216: 1.0}
    _times(monkeypatch, ms)
    table = autotune.tune(_instances(), cache_path=None)
    assert [c for _, _, c in probes] == list(autotune.CANDIDATES) and 0 in autotune.CANDIDATES
    for n, branches, _ in probes:
        assert n >= 2 and branches >= 2
    # as wide as 608 CTAs: kept against it, and against a wider one as fast
    assert list(table.values())[0]["ctas"] == 0


def test_narrower_tiling_within_the_slack_is_kept(probes, monkeypatch):
    _times(monkeypatch, {0: 1.0, 76: 1.3, 152: 1.08, 304: 1.01, 608: 1.02, 1216: 1.0})
    assert list(autotune.tune(_instances(), cache_path=None).values())[0]["ctas"] == 152


def test_cache_of_another_library_is_timed_again(probes, monkeypatch, tmp_path):
    path = str(tmp_path / "tune.json")
    _times(monkeypatch, {c: 1.0 for c in autotune.CANDIDATES})
    key = autotune.bucket(_instances()[0])
    stale = {key: {"ctas": 1216, "probe_ms": {}}}
    for content in (stale, {"library": "other", "table": stale}):
        with open(path, "w") as fh:
            json.dump(content, fh)
        n = len(probes)
        assert autotune.tune(_instances(), cache_path=path)[key]["ctas"] == 76
        assert len(probes) > n
    n = len(probes)
    assert autotune.tune(_instances(), cache_path=path)[key]["ctas"] == 76   # from the cache
    assert len(probes) == n
