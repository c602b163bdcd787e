"""Velocities whose FP32 parts are subnormal come back as they were given: the
state's conversions hold them exactly, and a set and a get without steps
between apply no arithmetic."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def test_subnormal_velocity_parts_survive_a_round_trip(mwlib):
    x, box = I.jittered_box(512, 1.0, 0.1, 8300)
    v = np.zeros((512, 3))
    rng = np.random.default_rng(8301)
    k = rng.integers(1, 1 << 20, size=(512, 3)).astype(np.float64)
    v[:200] = k[:200] * 2.0 ** -149 * rng.choice([-1.0, 1.0], size=(200, 3))  # subnormal leading parts
    v[200:400] = 2.0 ** -100 * (1.0 + 2.0 ** -40)  # a subnormal low part, 2^-140
    v[400:, 0] = 1e-3
    v[400:] = v[400:].astype(np.float32)
    s = mwlib.System(512, box)
    try:
        s.set_state(x, v)
        _, vg = s.get_state()
    finally:
        s.close()
    assert np.array_equal(vg, v)
