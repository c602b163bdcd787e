"""The grid-wide persistent engine on both sides of the number of boxes whose
thermostats every block evaluates for itself (8), against the oracle.  The
phase marks keep small systems on that engine.  FP32 forces grow to about 1e-5
A after 20 steps; 5e-5 allowed, as for the other engines."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [1, 2])  # Berendsen, Nose-Hoover
@pytest.mark.parametrize("nbox", [1, 8, 9])
def test_boxes_match_oracle(mwlib, orc, nbox, kind):
    xs, vs, boxes, T = [], [], [], []
    sizes = [216 + 13 * k for k in range(nbox)]
    for k, n in enumerate(sizes):
        x, b = I.jittered_box(n, 0.95 + 0.01 * k, 0.1, 300 + k)
        xs.append(I.snap_to_grid(x, b))
        boxes.append(b)
        T.append(230.0 + 10.0 * k)
        vs.append(I.maxwell_velocities(n, 1.2 * T[-1], seed=400 + k))
    s = mwlib.System(sizes, np.array(boxes))
    try:
        s.set_engine(mwlib.MW_ENGINE_PERSISTENT)
        s.set_phase_marks(1)
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        for steps in (1, 4, 7):
            th = s.step(steps, dt=10.0, thermostat=kind, T0_per_box=T, tau=200.0)
        xg, _ = s.get_state()
    finally:
        s.close()
    off = np.concatenate([[0], np.cumsum(sizes)])
    for k in range(nbox):
        xo, _, st, tho = orc.md(xs[k], vs[k], boxes[k], 12, dt=10.0, kind=kind, T0=T[k], tau=200.0)
        d = xg[off[k]:off[k + 1]] - xo
        assert np.abs(d - boxes[k] * np.rint(d / boxes[k])).max() < 5e-5
        assert th[k]["step"] == 12
        assert th[k]["pe"] == pytest.approx(tho[-1, 0], rel=3e-6)
        assert th[k]["ke"] == pytest.approx(tho[-1, 3], rel=1e-5)
        assert th[k]["xi"] == pytest.approx(st[0], rel=1e-4, abs=1e-9)


@pytest.mark.parametrize("steps", [100000, 100001])  # one launch; two
def test_long_asynchronous_runs(mwlib, steps):
    """Three atoms out of each other's reach, with one velocity: a straight line."""
    box = np.array([40.0, 41.0, 42.0])
    x = np.array([[1.0, 2.0, 3.0], [11.0, 2.0, 3.0], [1.0, 22.0, 3.0]])
    v = np.tile([2.0e-4, 0.0, -1.0e-4], (3, 1))
    s = mwlib.System(3, box)
    try:
        s.set_engine(mwlib.MW_ENGINE_PERSISTENT)
        s.set_state(x, v)
        mwlib.mw_step_async(s.h, mwlib.make_integrator(10.0, mwlib.MW_NVE, 300.0, 1000.0), steps)
        mwlib.mw_sync(s.h)
        assert s.thermo()[0]["step"] == steps
        xg, vg = s.get_state()
    finally:
        s.close()
    d = xg - (x + v * 10.0 * steps)
    # each step's move is rounded to FP32 (relative 6e-8): below 200 A * 6e-8
    assert np.abs(d - box * np.rint(d / box)).max() < 2e-5
    assert np.abs(vg - v).max() < 1e-12
