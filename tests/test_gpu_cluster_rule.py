"""The form that mw_step's persistent engine takes by size, where both were
measured: clusters where they are the faster form, the grid-wide form for few
large boxes and for batches just past what the chip holds at a time."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nbox,n,thermostat,clustered", [
    (1, 512, 0, True), (1, 1000, 2, False), (4, 1000, 2, True), (4, 3000, 2, False), (8, 4096, 3, True),
    (16, 1000, 2, True), (24, 4096, 2, True), (45, 500, 3, True), (64, 1000, 2, True), (200, 500, 2, True),
    (40, 4000, 3, False), (80, 2000, 3, False),
])
def test_form_by_size(mwlib, nbox, n, thermostat, clustered):
    x, box = I.jittered_box(n, 1.0, 0.1, 8800)
    s = mwlib.System([n] * nbox, np.tile(box, (nbox, 1)))
    try:
        s.set_engine(2)
        s.set_state(np.tile(x, (nbox, 1)))
        s.step(2, dt=5.0, thermostat=thermostat, T0=200.0)
        assert (s.info()["cluster_blocks"] > 0) == clustered
        if (nbox, n) == (200, 500):
            assert s.info()["cluster_blocks"] == 2
    finally:
        s.close()
