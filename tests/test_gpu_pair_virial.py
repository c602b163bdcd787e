"""The pair part of the virial where the three-body weight of a leg is zero:
lambda = 0 (accepted: pairs alone), or gamma so large that exp(gamma sigma /
(r - a sigma)) underflows well inside the cutoff.  Every force kernel against
the oracle, tolerances as in test_gpu_parity.py; for several species 1e-5 of
virial_abs as in test_gpu_species.py."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

from _parity import compare

pytestmark = pytest.mark.gpu

PARAMS = {"lambda_0": ("lambda_", "lambda", 0.0), "gamma_30": ("gamma", "gamma", 30.0)}
SHAPES = {"4x8": (4, 8, 0), "2x8": (2, 8, 0), "8x8": (8, 8, 0), "owner": (4, 8, 1)}


def _case(mwlib, orc, which):
    x, box = I.jittered_box(1000, 1.0, 0.25, 8200)
    x = I.snap_to_grid(x, box)
    field, name, value = PARAMS[which]
    prm = mwlib.mw_params_default()
    setattr(prm, field, value)
    return x, box, prm, orc.params(**{name: value})


@pytest.mark.parametrize("path", sorted(SHAPES) + ["plain"])
@pytest.mark.parametrize("which", sorted(PARAMS))
def test_pair_virial_of_every_force_kernel(mwlib, orc, which, path):
    x, box, prm, po = _case(mwlib, orc, which)
    s = mwlib.System(len(x), box, prm)
    try:
        if path == "plain":
            s.set_engine(mwlib.MW_ENGINE_PLAIN)
        else:
            mwlib.mw_set_force_shape(s.h, *SHAPES[path])
        s.set_state(x)
        f, e, w = s.energy_forces()
    finally:
        s.close()
    ref = orc.energy_forces(x, box, po)
    assert np.abs(ref["virial"][:3]).min() > 1e-2 * ref["virial_abs"]
    compare(f"{which} [{path}]", f, e[0], w[0], ref)


@pytest.mark.parametrize("grid_wide", [False, True])
@pytest.mark.parametrize("which", sorted(PARAMS))
def test_pair_virial_of_the_persistent_engine(mwlib, orc, which, grid_wide):
    """The record's virial after two steps: the oracle's at the same positions
    (the FP64 master positions differ from the 2^-32 grid by 3e-9 A at most)."""
    x, box, prm, po = _case(mwlib, orc, which)
    v = I.maxwell_velocities(len(x), 200.0, seed=8201)
    # four boxes: the cluster form's range
    s = mwlib.System([len(x)] * 4, np.tile(box, (4, 1)), prm)
    try:
        s.set_engine(2)
        if grid_wide:
            s.set_phase_marks(1)
        s.set_state(np.tile(x, (4, 1)), np.tile(v, (4, 1)))
        th = s.step(2, dt=10.0)
        xg, _ = s.get_state()
        assert (s.info()["cluster_blocks"] == 0) == grid_wide
    finally:
        s.close()
    for b in range(4):
        ref = orc.energy_forces(xg[b * len(x):(b + 1) * len(x)], box, po)
        assert np.abs(np.array(th[b]["virial"]) - ref["virial"]).max() <= 1e-6 * ref["virial_abs"], b


@pytest.mark.parametrize("kind", ["moments", "pairs"])
def test_pair_virial_of_several_species_with_a_large_gamma(mwlib, orc, kind):
    x, box = I.jittered_box(1000, 1.0, 0.25, 8202)
    x = I.snap_to_grid(x, box)
    t = (I.species_table_sw_family() if kind == "moments" else I.species_table_mixed(2, 5)).copy()
    t[..., 4] = 30.0  # gamma
    ty = I.species_draw(1000, len(t), 8203)
    s = mwlib.System(1000, box)
    try:
        s.set_species(t, ty)
        s.set_state(x)
        _, _, w = s.energy_forces()
        assert s.info()["species_moments"] == (1 if kind == "moments" else 0)
    finally:
        s.close()
    ref = orc.energy_forces_species(x, box, ty, t)
    assert np.abs(w[0] - ref["virial"]).max() <= 1e-5 * ref["virial_abs"]
