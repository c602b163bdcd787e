"""The grid-wide persistent engine's list builds on both sides of the limit
of its shared-memory scan (6144 cells), against the oracle's trajectory.  The
phase marks keep small systems on that engine."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I
from test_gpu_neighbors import _gas

pytestmark = pytest.mark.gpu

RL = 4.3065 + 0.3


@pytest.mark.parametrize("nc", [(4, 5, 6), (16, 16, 24), (18, 18, 19), (1, 1, 1)])  # 120, 6144, 6156 cells; a liquid
def test_builds_match_oracle(mwlib, orc, nc):
    if nc == (1, 1, 1):  # (18^3 atoms: about 19^3 cells of a short list radius, every cell occupied)
        x, box = I.jittered_box(5832, 1.0, 0.1, 21)
    else:
        x, box = _gas(300, [(c + 0.2) * RL for c in nc], 20)
    x = I.snap_to_grid(x, box)
    v = I.maxwell_velocities(len(x), 300.0, seed=22)
    s = mwlib.System(len(x), box, skin=0.3)
    try:
        s.set_engine(mwlib.MW_ENGINE_PERSISTENT)
        s.set_phase_marks(1)
        s.set_state(x, v)
        th = s.step(12, dt=10.0, thermostat=2, T0=300.0, tau=500.0)[0]
        assert th["rebuilds"] >= 4
        xg, _ = s.get_state()
    finally:
        s.close()
    xo, _, _, tho = orc.md(x, v, box, 12, dt=10.0, kind=2, T0=300.0, tau=500.0)
    d = xg - xo
    assert np.abs(d - box * np.rint(d / box)).max() < 5e-5
    assert abs(th["pe"] - tho[-1, 0]) <= 3e-6 * abs(tho[-1, 0])
