"""Single-point calls on a system that is in the middle of something: new
device positions while a half-kick is pending, a refused input, and cell
counts on both sides of the one-block scan's limit (8192)."""
import numpy as np
import pytest

from paper_0809_2811_gb300 import inputs as I
from _parity import F_TOL, force_err
from test_gpu_neighbors import R, _gas
from test_gpu_parity import check_neighbors

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [[700], [216, 500, 333]])
def test_positions_given_while_a_half_kick_is_pending(mwlib, orc, n):
    """mw_energy_forces_dev with new positions after a step: forces and
    energies of those positions, and the velocities are the step's (its
    closing half-kick taken with the old forces)."""
    torch = pytest.importorskip("torch")
    xs, vs, boxes, xn = [], [], [], []
    for k, m in enumerate(n):
        x, b = I.jittered_box(m, 1.0, 0.15, 9500 + k)
        xs.append(I.snap_to_grid(x, b))
        boxes.append(b)
        vs.append(I.maxwell_velocities(m, 280.0, seed=9600 + k))
        xn.append(I.snap_to_grid(I.jittered_box(m, 1.0, 0.3, 9700 + k)[0], b))
    N = sum(n)
    s = mwlib.System(n, np.array(boxes))
    try:
        s.set_state(np.concatenate(xs), np.concatenate(vs))
        s.step(3, dt=10.0)
        _, v_before = s.get_state()
        xd = torch.from_numpy(np.concatenate(xn)).cuda()
        f = torch.full((N, 3), float("nan"), dtype=torch.float32, device="cuda")
        e = torch.full((len(n), 3), float("nan"), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        mwlib.mw_energy_forces_dev(s.h, xd, f, e, None)
        _, v_after = s.get_state()
        # a non-finite position: refused, outputs untouched
        bad = xd.clone()
        bad[N // 2, 1] = float("inf")
        keep = f.clone()
        torch.cuda.synchronize()
        with pytest.raises(mwlib.MWError) as err:
            mwlib.mw_energy_forces_dev(s.h, bad, f, e, None)
        assert err.value.status == mwlib.MW_EINVAL and torch.equal(f, keep)
    finally:
        s.close()
    assert np.abs(v_after - v_before).max() <= 1e-15 + 1e-13 * np.abs(v_before).max()
    off = 0
    for k, m in enumerate(n):
        ref = orc.energy_forces(xn[k], boxes[k])
        assert force_err(keep[off:off + m].cpu().numpy(), ref["forces"]) <= F_TOL
        assert abs(float(e[k, 0]) - ref["energy"]) <= 1e-6 * (abs(ref["e2"]) + abs(ref["e3"]))
        off += m


@pytest.mark.parametrize("nc", [(20, 20, 20), (16, 16, 32), (21, 20, 20)])  # 8000, 8192, 8400 cells
def test_scan_limits(mwlib, orc, nc):
    x, box = _gas(300, [(c + 0.3) * R for c in nc], 11)
    x = I.snap_to_grid(x, box)
    s = mwlib.System(len(x), box)
    try:
        s.set_state(x)
        s.build_neighbors()
        assert s.info()["ncell_total"] == nc[0] * nc[1] * nc[2]
        check_neighbors(s, orc, x, box)
    finally:
        s.close()
