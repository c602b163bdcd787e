"""Positions into the 64-bit box fractions and back, where the integer
conversions could go wrong: many edges away, negative, next to a face, on it,
tiny; one box and several of different edges in one block.  A position comes
back as x - L floor(x / L) to a few FP64 ulp of its largest part, unwrapped as
given, and positions on the 2^-32 grid of the box exactly."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _positions(L, seed):
    rng = np.random.default_rng(seed)
    u = rng.uniform(0.0, 1.0, (40, 3))
    x = [u * L, -u * L, (u + 3.0) * L, (u - 1000.0) * L, (u - 0.5) * 1e9 * L, u * 1e-9 * L, -u * 1e-9 * L,
         u * 1e-25, -u * 1e-25, np.rint(8 * u - 4) * L, np.nextafter(np.broadcast_to(L, (40, 3)), 0.0), np.zeros((40, 3))]
    return np.concatenate(x)


@pytest.mark.parametrize("edges", [[[31.7, 12.9, 450.3]], [[12.0, 13.0, 14.0], [23.7, 17.1, 11.3], [60.0, 11.0, 29.9]]])
def test_round_trip(mwlib, edges):
    xs = [_positions(np.array(e), 30 + k) for k, e in enumerate(edges)]
    n = [len(x) for x in xs]
    x, L = np.concatenate(xs), np.repeat(np.array(edges), n, 0)
    s = mwlib.System(n, np.array(edges))
    try:
        s.set_state(x, np.zeros_like(x))
        got, _ = s.get_state()
        un = s.get_unwrapped()
    finally:
        s.close()
    tol = 4.0 * np.finfo(float).eps * np.maximum(np.abs(x), L)
    d = got - (x - L * np.floor(x / L))
    d -= L * np.rint(d / L)  # either side of a face
    assert (np.abs(d) <= tol).all()
    assert (got >= 0.0).all() and (got <= L).all()
    near = np.abs(x) < 2.0 ** 31 * L * 0.99  # (image counts are 32-bit)
    assert (np.abs(un - x)[near] <= tol[near]).all()


def test_grid_positions_exactly(mwlib):
    box = np.array([31.7, 44.4, 452.9])
    rng = np.random.default_rng(40)
    x = I.snap_to_grid(rng.uniform(0.0, 1.0, (3000, 3)) ** 6 * box, box)
    s = mwlib.System(len(x), box)
    try:
        s.set_state(x, None)
        got, _ = s.get_state()
    finally:
        s.close()
    assert np.array_equal(got, x)
