"""Asynchronous runs queued behind one that failed do nothing: the state stays
at the failing step, and mw_sync reports the first failure."""
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("thermostat", [0, 2])
def test_run_queued_behind_a_timed_out_one_does_nothing(mwlib, thermostat):
    x, v, box = I.nve512()
    it = mwlib.make_integrator(10.0, thermostat, 300.0, 1000.0)
    s = mwlib.System(512, box)
    try:
        s.set_engine(2)
        s.set_state(x, v)
        s.step(3, dt=10.0, thermostat=thermostat, T0=300.0, tau=1000.0)
        s.set_wait_limit(0.0)  # the next launch's first grid barrier gives up at once
        mwlib.mw_step_async(s.h, it, 5)
        s.set_wait_limit(2.0)
        mwlib.mw_step_async(s.h, it, 40)
        with pytest.raises(mwlib.MWError) as ei:
            mwlib.mw_sync(s.h)
        assert ei.value.status == mwlib.MW_ETIMEOUT
        assert s.thermo()[0]["step"] < 3 + 5
        s.set_state(x, v)
        assert s.step(4, dt=10.0)[0]["step"] == 4
    finally:
        s.close()


def _collapsing(mwlib):
    x, box = I.jittered_box(512, 0.80, 0.25, 901)
    x = I.snap_to_grid(x, box)
    v = I.maxwell_velocities(512, 250.0, seed=902)
    it = mwlib.make_integrator(10.0, mwlib.MW_NPT, 250.0, 200.0, p_ext=0.0, tau_p=500.0)
    s = mwlib.System(512, box)
    s.set_engine(2)
    s.set_state(x, v)
    mwlib.mw_step(s.h, it, 0, 1)
    return s, it


def test_isobaric_run_queued_behind_one_that_left_its_grid_does_nothing(mwlib):
    done = []
    for queued in (1, 2):
        s, it = _collapsing(mwlib)
        try:
            for _ in range(queued):
                mwlib.mw_step_async(s.h, it, 15)  # (leaves its grid within these)
            with pytest.raises(mwlib.MWError) as ei:
                mwlib.mw_sync(s.h)
            assert ei.value.status == mwlib.MW_EGRID
            done.append(s.thermo()[0]["step"])
            assert done[-1] < 15
            mwlib.mw_step_async(s.h, it, 30 - done[-1])
            mwlib.mw_sync(s.h)
            assert s.thermo()[0]["step"] == 30
        finally:
            s.close()
    assert done[0] == done[1]
