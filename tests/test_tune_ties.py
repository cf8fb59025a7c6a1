"""Which timings the tile tuner takes as ties, and which cached ones it trusts (no GPU)."""

import json

import pytest

from paper_1712_07973_gb300 import tune


# (ms per call by tile edge, choice): the fastest wherever a call's time is told
# apart from the scatter of its launches, however small the share; else the larger
@pytest.mark.parametrize("timings,best", [
    ({6: 28.6, 8: 31.2}, 6), ({6: 31.2, 8: 31.3}, 6), ({4: 4.49, 8: 4.50}, 4), ({2: 0.9, 6: 0.300, 8: 0.310}, 6),
    ({6: 0.0425, 8: 0.0426}, 8), ({6: 0.0414, 8: 0.0449}, 8), ({4: 0.050, 6: 0.0425, 8: 0.0500}, 6),
    ({6: 1.0, 8: 1.005}, 8), ({6: 1.0, 8: 1.007}, 6),
])
def test_ties_are_the_scatter_of_short_calls(timings, best):
    assert tune.select(timings) == best


def test_tiles_timed_on_other_kernels_are_not_reused(tmp_path, monkeypatch):
    path = str(tmp_path / "tiles.json")
    monkeypatch.setattr(tune, "_sm_count", lambda: 152)
    key = tune.cache_key(96, 64, "fp32", 152)
    with open(path, "w") as fh:  # as written before entries named their kernels
        json.dump({key: {"tile": 4, "ms": {"4": 1.0, "8": 2.0}}}, fh)
    assert tune.best_tile(96, 64, "fp32", path=path) == 0
    tune.tune(96, 64, "fp32", path=path, measure=lambda t: 9.0 - t, sm_count=152)
    assert tune.best_tile(96, 64, "fp32", path=path) == 8
    d = json.load(open(path))
    d[key]["kernels"] = "other"
    json.dump(d, open(path, "w"))
    assert tune.best_tile(96, 64, "fp32", path=path) == 0
