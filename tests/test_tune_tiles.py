"""The tile-column autotuner's choice (Solver.tune_tiles): the fastest candidate
where the per-phase kernels run, and the size rule (0) where the persistent
kernel runs, whose steps have no tile columns. Host logic, with the steps'
times made up."""
import time

import pytest

from paper_2303_10499_gb300 import gea


@pytest.mark.parametrize("driver,best", [("graph", 4), ("mixed", 4), ("persistent", 0), ("mixed_persistent", 0)])
def test_choice_by_driver(monkeypatch, driver, best):
    s = gea.Solver.__new__(gea.Solver)
    s.h = None
    cost = {1: 3e-3, 4: 1e-3, 8: 2e-3}
    seen = {"tiles": [], "steps": 0, "t": 0.0}

    def step(n=1):
        seen["steps"] += n
        seen["t"] += n * cost[seen["tiles"][-1]]
    monkeypatch.setattr(s, "stats", lambda: {"driver": driver}, raising=False)
    monkeypatch.setattr(s, "set_tiles_per_block", lambda n: seen["tiles"].append(n), raising=False)
    monkeypatch.setattr(s, "step", step, raising=False)
    monkeypatch.setattr(time, "perf_counter", lambda: seen["t"])
    res = s.tune_tiles(candidates=tuple(cost), steps=3)
    assert res["tiles_per_block"] == seen["tiles"][-1] == best
    assert set(res["ms_per_step"]) == set(cost) and seen["steps"] == 4 * len(cost)
