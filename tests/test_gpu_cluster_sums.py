"""The cluster form's kinetic energy is summed in FP64 beyond a warp.

Atoms 5 A apart (no forces), with speeds a 2^-17 A/fs, 256 <= a < 512, and a
mass of 2^14 times 4.184e-4 g/mol, so that an atom's kinetic energy is
a^2 2^-21 exactly and a warp's 32 of them (below 2^23 units of 2^-21) add up
exactly in FP32.  The total of 700 atoms is then exact if and only if nothing
above a warp is rounded to FP32.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KFCONV = 4.184e-4  # (kcal/mol/A)/(g/mol) -> A/fs^2


def test_kinetic_energy_is_exact_beyond_a_warp(mwlib):
    n, nbox, side = 700, 150, 9
    g = np.arange(side) * 5.0
    x0 = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)[:n] + 2.0
    rng = np.random.default_rng(8100)
    a = rng.integers(256, 512, size=(nbox, n))
    sign = rng.choice([-1.0, 1.0], size=(nbox, n))
    v = np.zeros((nbox, n, 3))
    axis = rng.integers(0, 3, size=(nbox, n))
    np.put_along_axis(v, axis[..., None], (sign * a * 2.0 ** -17)[..., None], axis=2)
    s = mwlib.System([n] * nbox, np.full((nbox, 3), 5.0 * side), mass=2.0 ** 14 * KFCONV)
    try:
        s.set_engine(2)
        s.set_state(np.tile(x0, (nbox, 1)), v.reshape(-1, 3))
        th = s.step(2, dt=1.0)
        assert s.info()["cluster_blocks"] in (1, 2)  # blocks of 350 atoms or more
    finally:
        s.close()
    want = (a.astype(np.int64) ** 2).sum(axis=1) * 2.0 ** -21
    got = np.array([t["ke"] for t in th])
    assert all(t["pe"] == 0.0 for t in th)
    assert np.array_equal(got, want), np.abs(got / want - 1).max()
