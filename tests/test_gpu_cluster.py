"""The persistent engine's cluster form (one thread-block cluster per box) at
the edges of its range, against the oracle's trajectories.

mw_step takes it for small boxes; the sizes below reach every cluster shape
(16, 8, 4, 2 and 1 blocks), blocks that hold no atom, last blocks that hold
one, a box with more cells than a block's shared memory holds, and a
neighbour-list overflow that stops the boxes of a batch on different steps.
Tolerances as for the other engines over such runs (test_gpu_dynamics.py):
FP32 forces grow to about 1e-5 A after 20 steps, 5e-5 allowed.
"""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu

STEPS, TAU = 12, 300.0


def _boxes(sizes, seed):
    xs, vs, boxes, T = [], [], [], []
    for k, n in enumerate(sizes):
        x, b = I.jittered_box(n, 0.95 + 0.02 * (k % 5), 0.1, seed + k)
        xs.append(I.snap_to_grid(x, b))
        boxes.append(b)
        T.append(220.0 + 15.0 * (k % 6))
        vs.append(I.maxwell_velocities(n, T[-1], seed=seed + 5000 + k))
    return xs, vs, boxes, T


def _check(orc, sizes, xs, vs, boxes, T, xg, th, steps, which):
    off = np.concatenate([[0], np.cumsum(sizes)])
    for k in which:
        xo, vo, st, tho = orc.md(xs[k], vs[k], boxes[k], steps, dt=10.0, kind=2, T0=T[k], tau=TAU)
        d = xg[off[k]:off[k + 1]] - xo
        assert np.abs(d - boxes[k] * np.rint(d / boxes[k])).max() < 5e-5, k
        assert th[k]["step"] == steps
        assert th[k]["pe"] == pytest.approx(tho[-1, 0], rel=3e-6)
        assert th[k]["ke"] == pytest.approx(tho[-1, 3], rel=1e-5)
        assert th[k]["xi"] == pytest.approx(st[0], rel=1e-4, abs=1e-9)


CASES = {
    "one_box_216": ([216], [0]),                       # 16 blocks of 14 atoms
    "one_box_1489": ([1489], [0]),                     # the last block short
    "uneven_6": ([1201, 217, 640, 999, 216, 512], [0, 1, 4]),
    "uneven_30": ([216 + 37 * k for k in range(30)], [0, 29]),   # 8 blocks
    "even_70": ([400] * 70, [0, 69]),                  # 4 blocks
    "even_150": ([256] * 150, [0, 149]),               # 2 blocks
    "even_300": ([216] * 300, [0, 299]),               # 1 block, more clusters than fit at once
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_cluster_trajectories_match_oracle(mwlib, orc, case):
    sizes, which = CASES[case]
    xs, vs, boxes, T = _boxes(sizes, 7000)
    s = mwlib.System(sizes, np.array(boxes))
    try:
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        s.step(STEPS - 5, dt=10.0, thermostat=2, T0_per_box=T, tau=TAU)  # (two runs: a pending half-kick between)
        th = s.step(5, dt=10.0, thermostat=2, T0_per_box=T, tau=TAU)
        xg, _ = s.get_state()
    finally:
        s.close()
    _check(orc, sizes, xs, vs, boxes, T, xg, th, STEPS, which)


def test_cluster_overflow_stops_boxes_on_their_own_steps(mwlib, orc):
    """Rows too narrow for some boxes: each box stops where its list overflows,
    the rows are grown, and every box finishes the run."""
    sizes = [300, 512, 216, 700, 450]
    xs, vs, boxes, T = _boxes(sizes, 7100)
    s = mwlib.System(sizes, np.array(boxes))
    try:
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        s.step(2, dt=10.0, thermostat=2, T0_per_box=T, tau=TAU)
        mwlib.mw_set_nbr_width(s.h, 6)
        th = s.step(STEPS - 2, dt=10.0, thermostat=2, T0_per_box=T, tau=TAU)
        xg, _ = s.get_state()
        again = s.step(3, dt=10.0, thermostat=2, T0_per_box=T, tau=TAU)
    finally:
        s.close()
    _check(orc, sizes, xs, vs, boxes, T, xg, th, STEPS, range(len(sizes)))
    assert all(t["step"] == STEPS + 3 for t in again)


def test_cluster_sparse_box_with_many_cells(mwlib, orc):
    """A droplet in a large cell: 30^3 = 27000 cells, more offsets than fit in
    a block's shared memory, so they are read back from global memory."""
    x, b = I.jittered_box(343, 1.0, 0.1, 7200)
    box = np.array([160.0, 161.0, 163.0])
    x = I.snap_to_grid(x + 60.0, box)
    v = I.maxwell_velocities(343, 250.0, seed=7201)
    s = mwlib.System(343, box, skin=0.3)  # a short skin: several list builds in the run
    try:
        s.set_state(x, v)
        th = s.step(STEPS, dt=10.0, thermostat=2, T0=250.0, tau=TAU)
        assert th[0]["rebuilds"] >= 3
        xg, _ = s.get_state()
    finally:
        s.close()
    _check(orc, [343], [x], [v], [box], [250.0], xg, th, STEPS, [0])
