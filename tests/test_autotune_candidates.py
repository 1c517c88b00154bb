"""The tuner times each launch once (CPU: the timing itself replaced)."""

import json

import pytest

from paper_2009_09500_gb300 import autotune, build, vox

BRICKS, RAGGED = (1024, 1024, 1024), (1000, 70, 33)


def setup_module(_):
    build.build_library()
    vox.load()


@pytest.mark.parametrize("dims,flags,timed", [
    (BRICKS, vox.OUT_LIST32, 3),                     # ctas_per_sm 0, 2, 4
    (BRICKS, vox.OUT_LIST64 | vox.OUT_BITMASK, 15),  # bricks with those, and 3 run lengths x 2 x 2 atomics
    (RAGGED, vox.OUT_BITMASK, 13),                   # atomics, and with 4 CTAs per SM
    (None, None, 19),                                # unknown: only list_runs has no effect
])
def test_each_launch_is_timed_once(monkeypatch, dims, flags, timed):
    in_force = []

    def measure(run, reps):
        in_force.append(vox.vox_get_tuning())
        return float(len(in_force))

    monkeypatch.setattr(autotune, "measure", measure)
    try:
        best, timings = autotune.tune(lambda: None, dims=dims, flags=flags)
    finally:
        vox.vox_reset_tuning()
    launches = [autotune.effective(t, dims, flags) for t in in_force]
    assert len(launches) == len(set(launches)) == len(timings) == timed
    assert set(launches) == {autotune.effective(c, dims, flags) for c in autotune.CANDIDATES}
    assert best == autotune.CANDIDATES[0] and json.dumps(best, sort_keys=True) in timings
