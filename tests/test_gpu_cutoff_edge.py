"""Pairs within an FP32 ulp or two of the cutoff a sigma.  For a quarter of all
sigmas some squared distance there has a square root that the hardware
approximation rounds to the cutoff itself, which made 1/(r - a sig) infinite
and the whole box's energy NaN; such a pair contributes nothing."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sigma", [2.3925, 2.9, 2.0015, 2.75, 3.1, 3.333])
def test_pairs_at_the_cutoff_are_finite(mwlib, sigma):
    rc = 1.8 * sigma
    n = 2048  # boxes of two atoms, in all directions so that every FP32 squared distance near the cutoff's is met
    rng = np.random.default_rng(5)
    u = rng.normal(size=(n, 3))
    u /= np.linalg.norm(u, axis=1)[:, None]
    r = rc * (1.0 + 2.0 ** -24 * rng.uniform(-8.0, 2.0, n))
    box = np.tile([40.0, 41.0, 42.0], (n, 1))
    x = np.zeros((2 * n, 3))
    x[0::2] = [10.0, 12.0, 13.0]
    x[1::2] = x[0::2] + r[:, None] * u
    p = mwlib.mw_params_default()
    p.sigma = sigma
    s = mwlib.System([2] * n, box)
    try:
        s.set_params(p)
        s.set_state(x)
        f, e, w = s.energy_forces()
    finally:
        s.close()
    # every term vanishes there faster than any power of the distance
    assert np.isfinite(f).all() and np.isfinite(e).all() and np.isfinite(w).all()
    assert np.abs(f).max() == 0.0 and np.abs(e).max() == 0.0
