"""The autotuner leaves pools alone whose streaming kernel takes several warps per cell: no launch shape applies
there, so its timings would differ by noise only, and a choice cached from them would be applied to later
solvers of the same size bucket (host logic, on a stand-in for the solver)."""
import json

import pytest


class _Solver:
    params = [{"precision": "fp32", "n_cells": 120}]
    n = 1

    def __init__(self, warps):
        self.warps, self.shape, self.timed = warps, (128, 1, 2), 0

    def launch(self):
        t, r, g = self.shape
        return {"threads": t, "reg_capped": r, "groups": g, "stream_warps": self.warps, "masked": 0, "heavy_min": 96,
                "ordered": 0}

    def set_launch(self, t, r, g):
        self.shape = (t, r, g)

    def step_timed(self, n):
        self.timed += n
        return [0.0, float(n) * (1.0 if self.shape == (64, 0, 3) else 2.0)] + [0.0] * 5, [0.0] * n


@pytest.fixture
def tuner(tmp_path, monkeypatch):
    from paper_2305_12071_gb300 import autotune
    monkeypatch.setattr(autotune, "_CACHE", str(tmp_path / "cache.json"))
    monkeypatch.setattr(autotune, "_key", lambda s: "key")
    return autotune


@pytest.mark.parametrize("warps", [2, 4, 8])
def test_no_shape_is_timed_or_cached_where_none_applies(tuner, tmp_path, warps):
    (tmp_path / "cache.json").write_text(json.dumps({"key": {"version": tuner._VERSION, "threads": 512, "reg_capped": 2,
                                                             "groups": 3}}))
    before = (tmp_path / "cache.json").read_text()
    s = _Solver(warps)
    assert tuner.tune(s) == ((128, 1, 2), {})
    assert s.timed == 0 and s.shape == (128, 1, 2) and (tmp_path / "cache.json").read_text() == before


def test_a_warp_per_cell_is_tuned_and_cached(tuner, tmp_path):
    # (an entry of an older version may come from a pool without a shape: not used)
    (tmp_path / "cache.json").write_text(json.dumps({"key": {"version": 3, "threads": 512, "reg_capped": 2, "groups": 3}}))
    s = _Solver(1)
    choice, timings = tuner.tune(s)
    assert choice == s.shape == (64, 0, 3) and len(timings) == len(tuner.CANDIDATES_FP32)
    t = _Solver(1)
    assert tuner.tune(t)[0] == t.shape == (64, 0, 3) and t.timed == 0
