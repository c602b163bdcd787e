"""MW_ENGINE_AUTO takes the engine that is the faster one by measurement: the
persistent engine up to a number of atoms that falls with the number of boxes
and lies higher without a thermostat."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu

NVE, NH, NPT = 0, 2, 3
CASES = [  # boxes, atoms a box, thermostat, engine (1 graph, 2 persistent)
    (1, 262144, NVE, 2), (1, 262144, NH, 2), (1, 262144, NPT, 2), (1, 350000, NH, 1), (1, 430000, NVE, 1),
    (9, 17777, NVE, 2), (9, 17777, NH, 2), (40, 7500, NH, 1), (130, 2000, NH, 1), (320, 500, NVE, 2),
    (145, 1000, NH, 2),
]


@pytest.mark.parametrize("nbox,n,thermostat,engine", CASES)
def test_engine_by_size_boxes_and_thermostat(mwlib, nbox, n, thermostat, engine):
    x, box = I.jittered_box(n, 1.0, 0.1, 8700)
    s = mwlib.System([n] * nbox, np.tile(box, (nbox, 1)))
    it = mwlib.make_integrator(5.0, thermostat, 200.0, 1000.0)
    try:
        s.set_state(np.tile(x, (nbox, 1)))
        s.step(1, dt=5.0, thermostat=thermostat, T0=200.0)
        assert s.info()["engine"] == engine
        mwlib.mw_step_async(s.h, it, 1)
        mwlib.mw_sync(s.h)
        assert s.info()["engine"] == engine
    finally:
        s.close()
