"""Neighbour sets of the list build at the edges of its two forms, bit-exact
against the oracle (outside the FP32/FP64 band of _parity.py): empty runs of
cells, exactly four cells on an axis (the shortest the packed form takes),
three and two (the wrapping form), cells at every face, and stencils of one
candidate more than a staging batch or a staging chunk holds."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I
from test_gpu_parity import check_neighbors

pytestmark = pytest.mark.gpu

R = 4.3065 + 1.0  # list radius at the default skin


def _gas(n, box, seed, dmin=2.2):
    """n atoms at random, no two closer than dmin (minimum image)."""
    rng = np.random.default_rng(seed)
    box = np.asarray(box, float)
    x = np.empty((0, 3))
    while len(x) < n:
        p = rng.uniform(0.0, 1.0, 3) * box
        d = x - p
        d -= box * np.rint(d / box)
        if not len(x) or (d * d).sum(1).min() > dmin * dmin:
            x = np.vstack([x, p])
    return x, box


CASES = {
    "gas_empty_runs": lambda: _gas(250, [40.0, 60.0, 80.0], 1),
    "four_cells_x": lambda: _gas(400, [4.05 * R, 5.1 * R, 6.2 * R], 2),
    "four_cells_all": lambda: _gas(300, [4.01 * R] * 3, 3),
    "three_cells_y": lambda: _gas(300, [5.0 * R, 3.2 * R, 4.4 * R], 4),
    "two_cells_z": lambda: _gas(200, [4.4 * R, 4.4 * R, 2.05 * R], 5),
    "corner_droplet": lambda: (I.jittered_box(257, 1.0, 0.2, 6)[0] - 9.0, np.array([64.0, 65.0, 66.0])),
    "chunk_edge": lambda: I.jittered_box(610, 1.26, 0.2, 7),  # ~257 candidates a stencil
    "batch_edge": lambda: I.jittered_box(700, 0.95, 0.2, 8),  # ~193
}


@pytest.mark.parametrize("case", sorted(CASES))
def test_neighbor_sets_match_oracle(mwlib, orc, case):
    x, box = CASES[case]()
    x = I.snap_to_grid(x, box)
    s = mwlib.System(len(x), box)
    try:
        s.set_state(x)
        s.build_neighbors()
        check_neighbors(s, orc, x, box)
    finally:
        s.close()
