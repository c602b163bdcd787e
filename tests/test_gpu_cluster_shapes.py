"""Every shape of the cluster form, asserted to have run: 1, 2, 4, 8 and 16
blocks per box, blocks full to the last thread (512 atoms), last blocks that
hold one atom and none, launches of two and three steps, isobaric boxes.
Trajectories against the oracle with the bounds of test_gpu_cluster.py (12
Nose-Hoover steps) and test_gpu_npt.py (its batch of three boxes, 15 steps)."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

from test_gpu_cluster import STEPS, TAU, _boxes, _check
from test_gpu_npt import _compare

pytestmark = pytest.mark.gpu

SIZES = {
    1: [512, 300],
    2: [1024, 513],
    4: [2048, 300],
    8: [4096, 57, 49],      # 8 atoms a block and one in the last; 7 a block and none in the last
    16: [8192, 241, 225],   # 16 and one; 15 and none
}


@pytest.mark.parametrize("blocks", sorted(SIZES))
def test_every_shape_matches_oracle(mwlib, orc, blocks):
    sizes = SIZES[blocks]
    xs, vs, boxes, T = _boxes(sizes, 8400)
    s = mwlib.System(sizes, np.array(boxes))
    try:
        s.set_engine(2)
        mwlib.mw_set_cluster_blocks(s.h, blocks)
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        done = 0
        while done < STEPS:
            k = min(2 + done % 3, STEPS - done)
            th = s.step(k, dt=10.0, thermostat=2, T0_per_box=T, tau=TAU)
            assert s.info()["cluster_blocks"] == (blocks if k > 1 else 0)
            done += k
        xg, _ = s.get_state()
    finally:
        s.close()
    _check(orc, sizes, xs, vs, boxes, T, xg, th, STEPS, range(len(sizes)))


@pytest.mark.parametrize("blocks", [1, 2, 4, 8, 16, -1])
def test_every_shape_isobaric_in_short_launches(mwlib, orc, blocks):
    n, rho, T = [216, 343, 290], [0.95, 1.0, 1.08], [230.0, 260.0, 300.0]
    xs, vs, boxes = [], [], []
    for k in range(3):
        x, b = I.jittered_box(n[k], rho[k], 0.2, 950 + k)
        xs.append(I.snap_to_grid(x, b))
        vs.append(I.maxwell_velocities(n[k], T[k], seed=960 + k))
        boxes.append(b)
    s = mwlib.System(n, np.array(boxes))
    try:
        s.set_engine(2)
        mwlib.mw_set_cluster_blocks(s.h, blocks)
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        for k in (2, 2, 2, 2, 2, 2, 3):
            th = s.step(k, dt=10.0, thermostat=mwlib.MW_NPT, T0_per_box=T, tau=300.0, p_ext=1.0, tau_p=1500.0)
            assert s.info()["cluster_blocks"] == max(blocks, 0)
        bg = s.box()
        xg, vg = s.get_state()
    finally:
        s.close()
    off = 0
    for k in range(3):
        xo, vo, bo, st, tho = orc.md_npt(xs[k], vs[k], boxes[k], 15, dt=10.0, T0=T[k], tau=300.0, p_atm=1.0,
                                         tau_p=1500.0)
        sl = slice(off, off + n[k])
        _compare(th[k], xg[sl], vg[sl], bg[k], xo, vo, bo, st, tho[-1], 15)
        off += n[k]


def test_shapes_that_do_not_fit_are_refused(mwlib):
    x, box = I.jittered_box(1025, 1.0, 0.1, 8500)
    s = mwlib.System(1025, box)
    try:
        for blocks in (1, 2, 3, 32, -2):
            with pytest.raises(mwlib.MWError) as ei:
                mwlib.mw_set_cluster_blocks(s.h, blocks)
            assert ei.value.status == mwlib.MW_EINVAL
        mwlib.mw_set_cluster_blocks(s.h, 4)
        s.set_engine(2)
        s.set_state(x)
        s.step(2, dt=10.0)
        assert s.info()["cluster_blocks"] == 4
        s.step(1, dt=10.0)
        assert s.info()["cluster_blocks"] == 0
        s.set_engine(1)
        s.step(2, dt=10.0)
        assert s.info()["cluster_blocks"] == 0
    finally:
        s.close()
