"""What a force call returns when the forces are valid already: the forces of
the last step of an isobaric run that left its cell grid on that step (a valid
step boundary), and the error of an asynchronous run that failed (its state is
not one to report forces of).  Tolerances as in test_gpu_parity.py."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

from _parity import compare

pytestmark = pytest.mark.gpu

KW = dict(dt=10.0, thermostat=3, T0=250.0, tau=200.0, p_ext=0.0, tau_p=500.0)


def _collapsing():
    """A liquid at 0.72 g/cm^3 under p = 0: its edge (27.71 A) is below the 5-cell grid's 26.53 A from step 3 on."""
    x, box = I.jittered_box(512, 0.72, 0.25, 901)
    return I.snap_to_grid(x, box), I.maxwell_velocities(512, 250.0, seed=902), box


def _system(mwlib, engine):
    x, v, box = _collapsing()
    s = mwlib.System(512, box)
    s.set_engine(1 if engine == "graph" else 2)
    if engine == "grid":
        s.set_phase_marks(1)  # (the cluster form records no marks: the grid-wide form runs)
    s.set_state(x, v)
    return s


def _leaving_step(mwlib):
    """The step at whose end the box has left its grid (laid out again when the run goes on)."""
    s = _system(mwlib, "graph")
    try:
        for k in range(1, 31):
            before = s.info()["regrids"]
            s.step(1, **KW)
            if s.info()["regrids"] > before:
                return k - 1
    finally:
        s.close()
    raise AssertionError("the box did not leave its grid")


@pytest.mark.parametrize("engine", ["graph", "grid", "cluster"])
def test_forces_of_the_step_that_left_the_grid(mwlib, orc, engine):
    torch = pytest.importorskip("torch")
    k = _leaving_step(mwlib)
    assert k >= 2
    s = _system(mwlib, engine)
    try:
        s.energy_forces()  # (other forces, energies and virials in the staging buffers)
        s.step(k, **KW)
        assert s.info()["regrids"] == 0
        assert (s.info()["cluster_blocks"] > 0) == (engine == "cluster")
        x, _ = s.get_state()
        box = s.box()[0]
        f, e, w = s.energy_forces()
        fd = torch.full((512, 3), float("nan"), dtype=torch.float32, device="cuda")
        ed = torch.full((1, 3), float("nan"), dtype=torch.float64, device="cuda")
        wd = torch.full((1, 6), float("nan"), dtype=torch.float64, device="cuda")
        mwlib.mw_energy_forces_dev(s.h, None, fd, ed, wd)
        s.step(1, **KW)
        assert s.info()["regrids"] == 1  # the run had left its grid on step k
    finally:
        s.close()
    ref = orc.energy_forces(x, box)
    compare(f"after the grid was left [{engine}]", f, e[0], w[0], ref)
    compare(f"after the grid was left [{engine}, device]", fd.cpu().numpy(), ed.cpu().numpy()[0], wd.cpu().numpy()[0], ref)


def test_asynchronous_force_call_after_the_grid_was_left(mwlib, orc):
    """mw_forces_async changes nothing until mw_sync has laid the grid out
    again; the forces, and the steps that take them, are those of the run."""
    k = _leaving_step(mwlib)
    x0, v0, box0 = _collapsing()
    s = _system(mwlib, "cluster")
    try:
        s.step(k, **KW)
        x, _ = s.get_state()
        box = s.box()[0]
        mwlib.mw_forces_async(s.h)
        with pytest.raises(mwlib.MWError) as ei:
            mwlib.mw_sync(s.h)
        assert ei.value.status == mwlib.MW_EGRID
        f, e, w = s.energy_forces()
        mwlib.mw_forces_async(s.h)
        mwlib.mw_sync(s.h)
        f2, _, _ = s.energy_forces()
        th = s.step(2, **KW)[0]
    finally:
        s.close()
    ref = orc.energy_forces(x, box)
    compare("asynchronous call, grid left", f, e[0], w[0], ref)
    compare("asynchronous call, grid laid out", f2, e[0], w[0], ref, force_only=True)
    _, _, bo, _, tho = orc.md_npt(x0, v0, box0, k + 2, dt=10.0, T0=250.0, tau=200.0, p_atm=0.0, tau_p=500.0)
    assert th["pe"] == pytest.approx(tho[-1, 0], rel=1e-6)  # as in test_gpu_npt.py
    assert th["ke"] == pytest.approx(tho[-1, 3], rel=3e-6)


@pytest.mark.parametrize("synced", [False, True])
def test_force_call_after_a_failed_asynchronous_run_reports_it(mwlib, synced):
    torch = pytest.importorskip("torch")
    x, v, box = I.nve512()
    it = mwlib.make_integrator(10.0, mwlib.MW_NVE)
    s = mwlib.System(512, box)
    try:
        s.set_engine(2)
        s.set_state(x, v)
        s.energy_forces()
        s.set_wait_limit(0.0)
        mwlib.mw_step_async(s.h, it, 5)
        s.set_wait_limit(2.0)
        if synced:
            with pytest.raises(mwlib.MWError) as ei:
                mwlib.mw_sync(s.h)
            assert ei.value.status == mwlib.MW_ETIMEOUT
        fd = torch.full((512, 3), 7.0, dtype=torch.float32, device="cuda")
        for call in (s.energy_forces, lambda: mwlib.mw_energy_forces_dev(s.h, None, fd)):
            with pytest.raises(mwlib.MWError) as ei:
                call()
            assert ei.value.status == mwlib.MW_ETIMEOUT
        assert bool((fd == 7.0).all())  # untouched after an error
        s.set_state(x, v)  # a new state: valid again
        s.energy_forces()
    finally:
        s.close()
