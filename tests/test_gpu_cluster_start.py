"""Many short launches of the persistent engine's cluster form: blocks without
atoms (216 atoms in blocks of 14 leave one of 16 empty) reach their first
exchange while others still load, and rank 0 sets the new edges of an isobaric
box at once.  Two steps a launch, against the oracle's trajectories; tolerances
as in test_gpu_npt.py."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

from test_gpu_npt import _compare

pytestmark = pytest.mark.gpu


def test_two_step_isobaric_launches_match_oracle(mwlib, orc):
    sizes, rho, T = [216, 230, 500, 217], [0.95, 1.0, 1.05, 0.98], [230.0, 260.0, 300.0, 250.0]
    xs, vs, boxes = [], [], []
    for k, n in enumerate(sizes):
        x, b = I.jittered_box(n, rho[k], 0.2, 7300 + k)
        xs.append(I.snap_to_grid(x, b))
        vs.append(I.maxwell_velocities(n, T[k], seed=7310 + k))
        boxes.append(b)
    s = mwlib.System(sizes, np.array(boxes))
    try:
        s.set_engine(2)
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        for _ in range(10):
            th = s.step(2, dt=10.0, thermostat=mwlib.MW_NPT, T0_per_box=T, tau=300.0, p_ext=1.0, tau_p=1500.0)
        bg = s.box()
        xg, vg = s.get_state()
    finally:
        s.close()
    off = np.concatenate([[0], np.cumsum(sizes)])
    for k in range(len(sizes)):
        xo, vo, bo, st, tho = orc.md_npt(xs[k], vs[k], boxes[k], 20, dt=10.0, T0=T[k], tau=300.0, p_atm=1.0,
                                         tau_p=1500.0)
        sl = slice(off[k], off[k + 1])
        _compare(th[k], xg[sl], vg[sl], bg[k], xo, vo, bo, st, tho[-1], 20)
