"""Runs without a thermostat, whose middle steps end after their forces: both
forms of the persistent engine against the oracle, and the errors that those
steps leave to the next one.  FP32 forces grow to about 1e-5 A after 20 steps;
5e-5 allowed, as for the other engines."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _system(mwlib, n, box, grid, **kw):
    s = mwlib.System(n, box, **kw)
    if grid:
        s.set_engine(mwlib.MW_ENGINE_PERSISTENT)
        s.set_phase_marks(1)  # keeps small systems on the grid-wide form
    return s


@pytest.mark.parametrize("grid", [False, True])
@pytest.mark.parametrize("runs", [(1, 2, 3, 6), (12,)])
def test_nve_matches_oracle(mwlib, orc, grid, runs):
    """A short skin (builds on quiet steps) and a row width that overflows after the first run."""
    sizes = [512, 343, 216]
    xs, vs, boxes = [], [], []
    for k, n in enumerate(sizes):
        x, b = I.jittered_box(n, 1.0, 0.1, 60 + k)
        xs.append(I.snap_to_grid(x, b))
        boxes.append(b)
        vs.append(I.maxwell_velocities(n, 280.0, seed=70 + k))
    s = _system(mwlib, sizes, np.array(boxes), grid, skin=0.3)
    try:
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        mwlib.mw_set_nbr_width(s.h, 6)
        for r in runs:
            th = s.step(r, dt=10.0)
        xg, vg = s.get_state()
    finally:
        s.close()
    off = np.concatenate([[0], np.cumsum(sizes)])
    for k in range(len(sizes)):
        xo, vo, _, tho = orc.md(xs[k], vs[k], boxes[k], 12, dt=10.0)
        d = xg[off[k]:off[k + 1]] - xo
        assert np.abs(d - boxes[k] * np.rint(d / boxes[k])).max() < 5e-5
        assert th[k]["step"] == 12 and th[k]["rebuilds"] >= 2
        assert th[k]["pe"] == pytest.approx(tho[-1, 0], rel=3e-6)
        assert th[k]["ke"] == pytest.approx(tho[-1, 3], rel=1e-5)


@pytest.mark.parametrize("grid", [False, True])
@pytest.mark.parametrize("gap", [0.02, 10.2])  # at once; 0.6 A apart after four steps
def test_colliding_atoms_are_reported(mwlib, grid, gap):
    x = np.array([[10.0, 10.0, 10.0], [10.0 + gap, 10.0, 10.0]] + [[5.0 + 4 * k, 25.0, 25.0] for k in range(5)])
    v = np.zeros_like(x)
    v[0, 0], v[1, 0] = 0.12, -0.12  # A / fs
    s = _system(mwlib, len(x), np.array([30.0, 31.0, 32.0]), grid)
    try:
        s.set_state(x, v)
        with pytest.raises(mwlib.MWError) as ei:
            s.step(40, dt=10.0)
        assert ei.value.status in (mwlib.MW_ENAN, mwlib.MW_ELOST)
    finally:
        s.close()
