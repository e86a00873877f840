"""Every plan search also times the library's own choice (no plan) and leaves
the grid or batch without a plan where that is as fast: synthetic timings, no
GPU."""
import json

import pytest

import paper_2002_12115_gb300.autotune as at
from paper_2002_12115_gb300 import JacError

DIMS = [(17, 33, 33), (33, 17, 33), (17, 17, 65)]
KD = (4, 8, 16)
SEARCHES = {
    "tune_batch": lambda b, path: at.tune_batch(b, passes=1, kdepths=KD, cache_path=path),
    "ga": lambda b, path: at.ga_tune_batch(b, M=4, T=3, kdepths=KD),
    "class_exhaustive": lambda b, path: at.class_exhaustive_tune_batch(b, kdepths=KD),
    "joint_exhaustive": lambda b, path: at.joint_exhaustive_tune_batch(b, kdepths=KD),
}


class StandInBatch:
    prec = "f32"

    def __init__(self):
        self.dims = DIMS
        self.plan = None
        self.measured = 0

    def set_plan(self, warps, tile_i, kdepth):
        self.plan = (warps, list(tile_i), list(kdepth))

    def sweep(self, n, residuals=True):
        pass

    def without_plan(self):
        return self.plan == (0, [0] * len(DIMS), [0] * len(DIMS))


class StandInGrid:
    prec, I, J, K = "f32", 65, 65, 65

    def __init__(self):
        self.plan = None
        self.measured = 0

    def set_plan(self, tile_j=0, kdepth=0, tile_i=0, fuse=0):
        if tile_j == 32:
            raise JacError(1, "unsupported plan")
        self.plan = (tile_j, kdepth, tile_i)

    def sweep(self, n):
        pass

    def without_plan(self):
        return self.plan == (0, 0, 0)


@pytest.fixture
def clock(monkeypatch):
    """time_call gives 1 s with a plan (a little more per tile column) and
    state["default"] without."""
    state = {"default": 0.5}

    def time_call(fn, reps=3, stream=None):
        x = state["on"]
        x.measured += 1
        if x.without_plan():
            return state["default"]
        tiles = x.plan[1] if isinstance(x.plan[1], list) else [x.plan[2]]
        return 1.0 + 1e-3 * sum(tiles)

    monkeypatch.setattr(at, "time_call", time_call)
    monkeypatch.setattr(at, "_gpu_name", lambda: "stand-in")
    return state


@pytest.mark.parametrize("search", SEARCHES)
@pytest.mark.parametrize("default", [0.5, 5.0])
def test_batch_keeps_the_faster_of_plan_and_none(clock, search, default):
    b = clock["on"] = StandInBatch()
    clock["default"] = default
    plan = SEARCHES[search](b, None)
    assert plan["no_plan"] == (default < 1.0) == b.without_plan()
    assert plan["warps"] in (4, 8) and set(plan["tile_i"]) == {"17", "33"}       # the search's own best
    n = 10 if search != "joint_exhaustive" else 5
    assert plan["default_s_per_sweep"] == default / n and plan["s_per_sweep"] > 1.0 / n
    if not plan["no_plan"]:
        assert b.plan[0] == plan["warps"] and b.plan[1] == [plan["tile_i"][str(d[0])] for d in DIMS]


@pytest.mark.parametrize("default", [0.5, 5.0])
def test_grid_keeps_the_faster_of_plan_and_none(clock, default, tmp_path):
    cache = str(tmp_path / "c.json")
    for _ in range(2):                                    # searched, then from the cache
        jac = clock["on"] = StandInGrid()
        clock["default"] = default
        best = at.tune_grid(jac, kdepths=(2, 8), cache_path=cache)
        assert best["no_plan"] == (default < 1.0) == jac.without_plan()
        assert best["tile_i"] == 16 and best["default_s_per_sweep"] == default / 20
    assert jac.measured == 0


def test_a_cached_decision_is_reused_and_older_entries_are_not(clock, tmp_path):
    cache = tmp_path / "c.json"
    b = clock["on"] = StandInBatch()
    first = SEARCHES["tune_batch"](b, str(cache))
    assert first["no_plan"]
    b = clock["on"] = StandInBatch()
    assert SEARCHES["tune_batch"](b, str(cache)) == first and b.measured == 0 and b.without_plan()
    # an entry of a search that did not time the library's choice
    old = {k.split("|", 1)[1]: {q: first[q] for q in ("warps", "tile_i", "kdepth", "s_per_sweep")}
           for k in json.loads(cache.read_text())}
    cache.write_text(json.dumps(old))
    b = clock["on"] = StandInBatch()
    assert SEARCHES["tune_batch"](b, str(cache))["no_plan"] and b.measured > 0 and b.without_plan()


def test_no_plan_ships_that_was_not_compared():
    """Entries of the cache beside the module, if it is there, carry the
    decision."""
    import os
    path = os.path.join(os.path.dirname(at.__file__), "autotune_cache.json")
    if os.path.exists(path):
        with open(path) as fh:
            assert all("no_plan" in v for v in json.load(fh).values())
