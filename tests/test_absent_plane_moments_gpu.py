"""Moment rows of FP64 bunches with Inf or NaN among their coordinates: the sums that contain them are
NaN, every other plane's are what they are without them, and a plane the bunch does not have stays
exactly 0 -- in each kind of kernel that holds all sixteen fields."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1610_05801_gb300 import phtl, synth  # noqa: E402

DEV = "cuda:0"
WIDE = dict(eta1=0.05, eta2=2.0, xi_x=5.0, xi_y=-3.0)
N = 60  # at most two blocks add to a row: their order does not matter


def _coords(bad):
    rng = np.random.default_rng(5)
    c = [rng.normal(0, s, N) for s in (0.1, 1e-3, 2e-3, 4e-5, 2e-3, 4e-5)]
    for i, v in bad.items():
        c[i][33] = v
    return c


def _rows(path, present, bad):
    ring = synth.ring(4.5e6, transverse=True, **(WIDE if path in ("widened", "rk4", "batch") else {}))
    bufs = [torch.tensor(a, dtype=torch.float64, device=DEV) if i // 2 in present else None
            for i, a in enumerate(_coords(bad))]
    mon = torch.zeros(2, phtl.MON_FIELDS, dtype=torch.float64, device=DEV)
    R = phtl.Ring(**ring)
    if path == "batch":
        B = phtl.Batch(R, [phtl.make_job(*bufs, turns=1, integrator="leapfrog", dtype="f64", monitor=mon)])
        B.run()
    else:
        R.set_monitor(mon, stride=1)
        if path == "ramp":
            R.set_programme(np.array([4.5e6]), np.array([26e9, 26e9 + 2e6]))
            R.track_programme(*bufs, turn0=0, turns=1, integrator="leapfrog")
        elif path == "collective":
            R.set_wake(np.exp(-np.arange(64.0) / 6), -0.75, 0.75, -5e-11, 1e-9)
            R.track_collective(*bufs, turns=1, integrator="leapfrog")
        else:
            R.track(*bufs, turns=1, integrator="rk4" if path == "rk4" else "leapfrog")
    torch.cuda.synchronize()
    if path == "batch":
        B.close()
    R.close()
    return mon.cpu().numpy()


@pytest.mark.parametrize("path", ["linear", "widened", "rk4", "ramp", "collective", "batch"])
@pytest.mark.parametrize("present", [(0,), (0, 1), (0, 2), (0, 1, 2)])
@pytest.mark.parametrize("bad", [{0: np.inf}, {1: np.nan}, {0: -np.inf, 1: np.inf}])
def test_non_finite_longitudinal_coordinates(path, present, bad):
    rows, clean = _rows(path, present, bad), _rows(path, present, {})
    assert np.all(rows[:, 0] == N)
    for plane in range(3):
        f = slice(1 + 5 * plane, 6 + 5 * plane)
        if plane not in present:
            assert np.all(rows[:, f] == 0.0), (plane, rows[:, f])
    # the initial row: only the fields with the bad coordinates are lost
    first = rows[0, 1:6]
    lost = [0 in bad, 1 in bad, 0 in bad, 1 in bad, True]
    assert np.all(np.isnan(first) == lost), first
    keep = ~np.array(lost)
    assert np.all(np.isfinite(first[keep]))
    assert np.array_equal(rows[0, 6:], clean[0, 6:])


@pytest.mark.parametrize("path", ["linear", "widened", "ramp"])
def test_non_finite_transverse_coordinate(path):
    rows, clean = _rows(path, (0, 1), {2: np.nan}), _rows(path, (0, 1), {})
    assert np.array_equal(rows[:, :6], clean[:, :6])
    assert np.all(np.isnan(rows[0, [6, 8, 10]])) and np.all(np.isfinite(rows[0, [7, 9]]))
    assert np.all(rows[:, 11:] == 0.0)
