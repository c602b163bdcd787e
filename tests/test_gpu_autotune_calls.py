"""The autotuner's choices for mw_step and mw_step_async where the persistent
engine's cluster form, which mw_step alone has, applies: mw_step's by what it
runs, mw_step_async's by what it runs, cached side by side; cache lines
without a choice for the asynchronous call hold for both."""
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu

T0, TAU = 260.0, 500.0


def _system(mwlib):
    x, box = I.jittered_box(512, 1.0, 0.1, 8600)
    v = I.maxwell_velocities(512, T0, seed=8601)
    s = mwlib.System(512, box)
    s.set_state(x, v)
    return s, mwlib.make_integrator(10.0, 2, T0, TAU)


def _engines(mwlib, s, it):
    mwlib.mw_step(s.h, it, 4, 1)
    a = s.info()
    mwlib.mw_step_async(s.h, it, 4)
    mwlib.mw_sync(s.h)
    b = s.info()
    assert b["cluster_blocks"] == 0
    return a["engine"], b["engine"], a["cluster_blocks"]


def test_each_call_gets_its_own_choice(mwlib, tmp_path, monkeypatch):
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("MW_AUTOTUNE_CACHE", str(path))
    s, it = _system(mwlib)
    try:
        mwlib.mw_set_cluster_blocks(s.h, 16)  # the cluster form applies
        best = mwlib.mw_autotune(s.h, it, 10)
        step, queued, blocks = _engines(mwlib, s, it)
        assert step == best and blocks == (16 if best == 2 else 0)
    finally:
        s.close()
    key, eng, skin, grid, shape, async_eng = path.read_text().split()
    assert (int(eng), int(async_eng)) == (step, queued)
    # cached choices, one per call
    for line, want in (((2, 1), (2, 1)), ((1, 2), (1, 2)), ((2,), (2, 2)), ((1,), (1, 1))):
        path.write_text(" ".join([key, str(line[0]), skin, "0", shape] + [str(k) for k in line[1:]]) + "\n")
        s, it = _system(mwlib)
        try:
            assert mwlib.mw_autotune(s.h, it, 10) == want[0]
            assert _engines(mwlib, s, it)[:2] == want
        finally:
            s.close()


def test_grid_sizes_of_a_clustered_batch_are_timed_as_the_asynchronous_call(mwlib, tmp_path, monkeypatch):
    """24 boxes of 600 atoms: the cluster form runs in mw_step; the cached grid
    is one of the two sizes that the grid-wide form was timed with."""
    import numpy as np
    path = tmp_path / "tune.txt"
    monkeypatch.setenv("MW_AUTOTUNE_CACHE", str(path))
    xs, vs, boxes = [], [], []
    for k in range(24):
        x, b = I.jittered_box(600, 1.0, 0.1, 8610 + k)
        xs.append(x)
        vs.append(I.maxwell_velocities(600, T0, seed=8640 + k))
        boxes.append(b)
    s = mwlib.System([600] * 24, np.array(boxes))
    it = mwlib.make_integrator(10.0, 2, T0, TAU)
    try:
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        mwlib.mw_autotune(s.h, it, 10)
        grid, async_eng = [int(k) for k in path.read_text().split()[3:6:2]]
        mwlib.mw_step_async(s.h, it, 3)
        mwlib.mw_sync(s.h)
        info = s.info()
        assert info["engine"] == async_eng
        assert grid == 0 or (async_eng == 2 and info["persistent_blocks"] == grid)
        s.step(4, dt=10.0, thermostat=2, T0=T0, tau=TAU)
        info = s.info()
        assert info["engine"] != 2 or info["cluster_blocks"] > 0
    finally:
        s.close()
