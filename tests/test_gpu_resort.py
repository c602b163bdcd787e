"""List builds that leave the atoms' order alone (all but every eighth of a
box's builds) against the oracle: trajectories long enough to pass several
builds of both kinds, then the neighbour sets, forces and states read back in
the caller's order.  Every engine, one box, a batch whose boxes build on
different steps, and two species (their types travel with the sort alone).
Tolerances as in test_gpu_dynamics.py."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I
from test_gpu_parity import check_neighbors

pytestmark = pytest.mark.gpu

ENGINES = {"graph": 1, "persistent": 2, "plain": 3}


@pytest.mark.parametrize("engine", sorted(ENGINES))
@pytest.mark.parametrize("n", [[300], [2500], [260, 700, 450]])
def test_many_builds_match_oracle(mwlib, orc, engine, n):
    xs, vs, boxes = [], [], []
    for k, m in enumerate(n):
        x, b = I.jittered_box(m, 1.0, 0.1, 9100 + k)
        xs.append(I.snap_to_grid(x, b))
        boxes.append(b)
        vs.append(I.maxwell_velocities(m, 250.0 + 20.0 * k, seed=9200 + k))
    s = mwlib.System(n, np.array(boxes), skin=0.25)  # a build nearly every step
    try:
        s.set_engine(ENGINES[engine])
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        th = s.step(20, dt=10.0, thermostat=2, T0=260.0, tau=400.0)
        assert min(t["rebuilds"] for t in th) > 9  # past the second sort
        xg, _ = s.get_state()
        f, _, _ = s.energy_forces()
    finally:
        s.close()
    off = 0
    for k, m in enumerate(n):
        xo, _, _, tho = orc.md(xs[k], vs[k], boxes[k], 20, dt=10.0, kind=2, T0=260.0, tau=400.0)
        d = xg[off:off + m] - xo
        assert np.abs(d - boxes[k] * np.rint(d / boxes[k])).max() < 5e-5
        assert th[k]["pe"] == pytest.approx(tho[-1, 0], rel=3e-6)
        fr = orc.energy_forces(np.mod(xg[off:off + m], boxes[k]), boxes[k])["forces"]
        assert np.abs(f[off:off + m] - fr).max() < 1e-5 * max(np.abs(fr).max(), 2.59)
        off += m


def test_sets_after_builds_without_a_sort(mwlib, orc):
    x, box = I.jittered_box(1000, 1.0, 0.1, 9300)
    s = mwlib.System(1000, box, skin=0.4)
    try:
        s.set_engine(mwlib.MW_ENGINE_GRAPH)
        s.set_state(x, I.maxwell_velocities(1000, 280.0, seed=9301))
        while True:  # to a step that has just built, without a sort (builds 2 to 8 of a box)
            before = s.thermo()[0]["rebuilds"]
            th = s.step(1, dt=10.0)[0]
            if th["rebuilds"] > before and th["rebuilds"] >= 3:
                break
        xg, _ = s.get_state()
        check_neighbors(s, orc, xg, box)
    finally:
        s.close()


def test_species_follow_their_atoms(mwlib, orc):
    x, box = I.jittered_box(1200, 0.9, 0.1, 9400)
    x = I.snap_to_grid(x, box)
    v = I.maxwell_velocities(1200, 260.0, seed=9401)
    types = I.species_draw(1200, 4, 5)
    table = I.species_table_sw_family()
    s = mwlib.System(1200, box, skin=0.25)
    try:
        s.set_species(table, types)
        s.set_state(x, v)
        th = s.step(20, dt=10.0)[0]
        assert th["rebuilds"] > 9
        xg, _ = s.get_state()
        f, e, _ = s.energy_forces()
    finally:
        s.close()
    r = orc.energy_forces_species(np.mod(xg, box), box, types, table)
    assert np.abs(f - r["forces"]).max() < 1e-5 * max(np.abs(r["forces"]).max(), 2.59)
    assert abs(e[0, 0] - r["energy"]) <= 1e-6 * (abs(r["e2"]) + abs(r["e3"]))
