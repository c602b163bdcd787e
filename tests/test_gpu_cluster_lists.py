"""Neighbour rows of boxes that had finished their steps when another box's
row overflowed (the cluster form grows the rows of all boxes), and rows given
up by mw_set_nbr_width or by a restored checkpoint while the forces stay valid:
every call that reads the rows builds them first.

170 boxes of 230 atoms at 0.95 g/cm^3 fit the given row width and fill the
device (largest boxes first); the 30 denser boxes that start when those have
finished do not.  Tolerances: forces 1e-5 and adjoint 1e-4 as in
test_gpu_parity.py and test_gpu_adjoint.py; neighbour sets exact outside the
FP32/FP64 band.
"""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

from _parity import F_TOL, force_err

pytestmark = pytest.mark.gpu

N_LOW, N_DENSE, LOW, DENSE = 230, 216, 170, 30
T0, TAU, STEPS = 240.0, 300.0, 8
KW = dict(dt=10.0, thermostat=2, T0=T0, tau=TAU)
WATCH = (0, 7, 101)  # boxes of the first wave


def _state():
    sizes = [N_LOW] * LOW + [N_DENSE] * DENSE
    xs, vs, boxes = [], [], []
    for k, n in enumerate(sizes):
        x, b = I.jittered_box(n, 0.95 if k < LOW else 1.7, 0.1, 7400 + k)
        xs.append(I.snap_to_grid(x, b))
        vs.append(I.maxwell_velocities(n, T0, seed=7800 + k))
        boxes.append(b)
    return sizes, np.concatenate(xs), np.concatenate(vs), np.array(boxes)


def _widest(mwlib, sizes, x, v, boxes, steps):
    s = mwlib.System(sizes, boxes)
    try:
        s.set_state(x, v)
        s.step(steps, **KW)
        return s.info()["max_count"]
    finally:
        s.close()


def _overflowed(mwlib):
    """A system after a run in which the dense boxes' rows overflowed."""
    sizes, x, v, boxes = _state()
    nl = LOW * N_LOW
    fit = _widest(mwlib, sizes[:LOW], x[:nl], v[:nl], boxes[:LOW], STEPS) + 3
    assert _widest(mwlib, sizes[LOW:], x[nl:], v[nl:], boxes[LOW:], 2) > fit
    s = mwlib.System(sizes, boxes)
    s.set_engine(2)
    s.set_state(x, v)
    s.step(0, **KW)
    mwlib.mw_set_nbr_width(s.h, fit)
    th = s.step(STEPS, **KW)
    assert all(t["step"] == STEPS for t in th)
    assert s.info()["nbr_width"] > fit  # the rows were grown during the run
    assert s.info()["cluster_blocks"] > 0
    return s, boxes


def _box_slices():
    return [slice(k * N_LOW, (k + 1) * N_LOW) for k in WATCH]


def test_neighbor_sets_after_cluster_overflow(mwlib, orc):
    s, boxes = _overflowed(mwlib)
    try:
        x, _ = s.get_state()
        info = s.info()
        counts, nbr = s.neighbors(width=info["max_count"])
    finally:
        s.close()
    for k, sl in zip(WATCH, _box_slices()):
        # every pair within the cutoff is listed (the list may be of earlier
        # positions of the run), nothing past the list radius plus the skin
        near, _ = orc.neighbors(x[sl], boxes[k], info["r_list"] - 1.0)
        far, _ = orc.neighbors(x[sl], boxes[k], info["r_list"] + 1.0)
        for i in range(N_LOW):
            c = counts[sl.start + i]
            got = set((nbr[sl.start + i, :c] - sl.start).tolist())
            assert len(got) == c, (k, i)
            assert set(near[i].tolist()) <= got <= set(far[i].tolist()), (k, i)


@pytest.mark.parametrize("forces_first", [False, True])
def test_adjoint_after_cluster_overflow(mwlib, orc, forces_first):
    torch = pytest.importorskip("torch")
    s, boxes = _overflowed(mwlib)
    try:
        x, _ = s.get_state()
        if forces_first:
            s.energy_forces()
        w = np.random.default_rng(5).normal(size=x.shape)
        wd = torch.tensor(w, dtype=torch.float32, device="cuda")
        gd = torch.zeros_like(wd)
        mwlib.mw_energy_forces_vjp(s.h, wd, gd, s.nbox)
        g = gd.cpu().numpy().astype(np.float64)
    finally:
        s.close()
    for k, sl in zip(WATCH, _box_slices()):
        ref, _ = orc.force_vjp(x[sl], boxes[k], w[sl])
        mag = np.linalg.norm(ref, axis=1)
        err = np.linalg.norm(g[sl] - ref, axis=1) / np.maximum(mag, np.sqrt(np.mean(mag ** 2)))
        assert err.max() <= 1e-4, k


def test_forces_async_and_steps_after_cluster_overflow(mwlib, orc):
    s, boxes = _overflowed(mwlib)
    try:
        x, v = s.get_state()
        mwlib.mw_forces_async(s.h)
        mwlib.mw_sync(s.h)
        f, _, _ = s.energy_forces()
        th = s.step(4, dt=10.0)
        x2, _ = s.get_state()
    finally:
        s.close()
    for k, sl in zip(WATCH, _box_slices()):
        assert force_err(f[sl], orc.energy_forces(x[sl], boxes[k])["forces"]) <= F_TOL, k
        xo, _, _, tho = orc.md(x[sl], v[sl], boxes[k], 4, dt=10.0)
        d = x2[sl] - xo
        assert np.abs(d - boxes[k] * np.rint(d / boxes[k])).max() < 5e-5, k
        assert th[k]["pe"] == pytest.approx(tho[-1, 0], rel=3e-6)


def test_rows_given_up_by_a_new_width_are_built_for_the_calls_that_read_them(mwlib, orc):
    torch = pytest.importorskip("torch")
    x, box = I.jittered_box(512, 1.0, 0.2, 7900)
    x = I.snap_to_grid(x, box)
    w = np.random.default_rng(6).normal(size=x.shape)
    ref_f = orc.energy_forces(x, box)["forces"]
    ref_g, _ = orc.force_vjp(x, box, w)
    s = mwlib.System(512, box)
    try:
        s.set_state(x)
        s.energy_forces()
        mwlib.mw_set_nbr_width(s.h, 64)
        wd = torch.tensor(w, dtype=torch.float32, device="cuda")
        gd = torch.zeros_like(wd)
        mwlib.mw_energy_forces_vjp(s.h, wd, gd, 1)
        g = gd.cpu().numpy().astype(np.float64)
        mwlib.mw_set_nbr_width(s.h, 96)
        mwlib.mw_forces_async(s.h)
        mwlib.mw_sync(s.h)
        f, _, _ = s.energy_forces()
    finally:
        s.close()
    mag = np.linalg.norm(ref_g, axis=1)
    assert (np.linalg.norm(g - ref_g, axis=1) / np.maximum(mag, np.sqrt(np.mean(mag ** 2)))).max() <= 1e-4
    assert force_err(f, ref_f) <= F_TOL


def test_rows_of_another_state_are_built_after_a_restore(mwlib, orc):
    torch = pytest.importorskip("torch")
    x, box = I.jittered_box(512, 1.0, 0.2, 7901)
    x = I.snap_to_grid(x, box)
    other = I.snap_to_grid(I.jittered_box(512, 1.0, 0.2, 7902)[0][::-1].copy(), box)
    w = np.random.default_rng(7).normal(size=x.shape)
    ref_g, _ = orc.force_vjp(x, box, w)
    s = mwlib.System(512, box)
    try:
        s.set_state(x)
        s.energy_forces()
        blob = s.checkpoint()
        s.set_state(other)
        s.energy_forces()
        s.restore(blob)
        wd = torch.tensor(w, dtype=torch.float32, device="cuda")
        gd = torch.zeros_like(wd)
        mwlib.mw_energy_forces_vjp(s.h, wd, gd, 1)
        g = gd.cpu().numpy().astype(np.float64)
    finally:
        s.close()
    mag = np.linalg.norm(ref_g, axis=1)
    assert (np.linalg.norm(g - ref_g, axis=1) / np.maximum(mag, np.sqrt(np.mean(mag ** 2)))).max() <= 1e-4
