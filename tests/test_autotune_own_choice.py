"""The tuner against the library's own choice (host logic, no GPU): a configuration names
the general kernel's launch, so nothing may be kept where the call without one is faster."""
import json

from paper_1409_0669_gb300 import autotune
from paper_1409_0669_gb300._native import LakCfg

CFGS = [LakCfg(64, 0, 1, 0), LakCfg(128, 0, 2, 0)]


class FakeProblem:
    nbytes = 10 ** 9
    op, storage = "gemv_row", "f32"
    # us of the two configurations and of the call without one, per size
    table = {100: (10.0, 11.0, 9.0), 200: (10.0, 12.0, 10.5), 900: (10.0, 9.0, 12.0)}

    def __init__(self, op, storage, size):
        self.us = self.table[size]
        self.dims = (size, size, 0)

    def time_cfg(self, cfg, reps):
        return self.us[2] if cfg is None else self.us[[c.block for c in CFGS].index(cfg.block)]


def test_own_choice_wins_its_bucket(monkeypatch):
    tune = autotune.tune
    monkeypatch.setattr(autotune, "Problem", FakeProblem)
    monkeypatch.setattr(autotune, "problem_bucket", lambda p: 1 if p.dims[0] < 500 else 2)
    monkeypatch.setattr(autotune.torch.cuda, "empty_cache", lambda: None)
    monkeypatch.setattr(autotune, "tune", lambda op, st, sz, reps, problem: tune(
        op, st, sz, reps, cfgs=CFGS, problem=problem))
    per = autotune.tune_buckets("gemv_row", "f32", [100, 200, 900])
    assert per[1]["cfg"] is None                  # 9/9 and 10/10.5, against 9/10 and 1
    assert abs(per[1]["worst_ratio"] - 10.0 / 10.5) < 1e-12
    assert per[2]["cfg"] == [128, 0, 2, 0] and per[2]["worst_ratio"] == 1.0


def test_ties_go_to_the_own_choice_and_none_leaves_the_cache(tmp_path, monkeypatch):
    res = {1: [{"cfg": [64, 0, 1, 0], "us": 5.0}]}
    assert autotune.choose_per_bucket(res, {1: 0}, {1: 5.0})[0]["cfg"] is None
    assert autotune.choose_per_bucket(res, {1: 0}, {1: 5.1})[0]["cfg"] == [64, 0, 1, 0]
    assert autotune.choose_per_bucket(res, {1: 0})[0]["cfg"] == [64, 0, 1, 0]
    monkeypatch.setattr(autotune, "cache_key", lambda: "GPU")
    path = tmp_path / "cache.json"
    autotune.save_cache(str(path), {"dot:f32:0": [64, 0, 1, 0], "dot:f32:1": [128, 0, 1, 0]})
    autotune.save_cache(str(path), {"dot:f32:1": None, "dot:f32:2": None})
    assert json.loads(path.read_text()) == {"GPU": {"dot:f32:0": [64, 0, 1, 0]}}
