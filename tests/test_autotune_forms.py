"""The autotuner compares launch shapes and layouts of a batch in one launch
form, and does not use tilings that were measured against other kernels (CPU,
with injected measurements)."""
import json

import pytest

from paper_1711_01919_gb300 import autotune, ihist

SHAPES = [(240, 320, 16), (480, 640, 32)]


def fake_time_batch(seen):
    def time_batch(shapes, tune, reps=3, tables=False, queries=0, replay=False):
        """Live, the untuned launch wins in quad-major; replayed, a tiling does in bin-major."""
        seen.append(replay)
        quad = shapes[0][3] == ihist.IHIST_QUAD_MAJOR
        if replay:
            return (6.0 if quad else 5.0) + (0.0 if tune.get("rows_per_band") == 40 else 1.0)
        return (4.0 if quad else 5.0) + (0.0 if tune == {} else 1.0)
    return time_batch


@pytest.mark.parametrize("replay,layout,tuned", [(False, ihist.IHIST_QUAD_MAJOR, False),
                                                 (True, ihist.IHIST_BIN_MAJOR, True)])
def test_layout_and_launch_shape_are_compared_in_the_callers_form(tmp_path, monkeypatch, replay, layout, tuned):
    monkeypatch.setenv("IHIST_TUNE_CACHE", str(tmp_path / "c.json"))
    seen = []
    monkeypatch.setattr(autotune, "time_batch", fake_time_batch(seen))
    got, tune, times = autotune.tune_batch_layout(SHAPES, device="fake", replay=replay)
    assert set(seen) == {replay}
    assert got == layout and bool(tune) == tuned and times[got] == min(times.values())


def test_live_and_replayed_launch_shapes_are_cached_apart(tmp_path, monkeypatch):
    monkeypatch.setenv("IHIST_TUNE_CACHE", str(tmp_path / "c.json"))
    seen = []
    monkeypatch.setattr(autotune, "time_batch", fake_time_batch(seen))
    batch = [s + (ihist.IHIST_BIN_MAJOR,) for s in SHAPES]
    for _ in range(2):
        assert autotune.tune_batch(batch, device="fake") == {}
        assert autotune.tune_batch(batch, device="fake", replay=True)["rows_per_band"] == 40
    n = len(autotune.batch_candidates(batch))
    assert seen == [False] * n + [True] * n  # the second round came from the cache


def test_tilings_measured_against_other_kernels_are_measured_again(tmp_path, monkeypatch):
    path = tmp_path / "c.json"
    monkeypatch.setenv("IHIST_TUNE_CACHE", str(path))
    batch = [s + (ihist.IHIST_BIN_MAJOR,) for s in SHAPES]
    old = {"rows_per_band": 64}

    def timer(t):
        return 1.0 if t == {} else 2.0

    plan_key = "plan|fake|480x640x32|0"
    autotune.tune_plan(480, 640, 32, timer=timer, device="fake")
    autotune.tune_batch(batch, timer=timer, device="fake")
    keys = list(json.load(open(path)))
    assert plan_key in keys and len(keys) == 2
    json.dump({k: {"tune": old, "ms": 0.5} for k in keys}, open(path, "w"))  # as an earlier library left them
    assert autotune.tune_plan(480, 640, 32, timer=timer, device="fake") == {}
    assert autotune.tune_batch(batch, timer=timer, device="fake") == {}
    assert autotune.tune_plan(480, 640, 32, timer=None, device="fake") == {}  # and kept
