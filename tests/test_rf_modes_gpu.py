"""FP64 kernels of each RF mode (phi_s or not, second RF system and slippage expansion or not,
rf_linear) against the oracle: each mode is a kernel of its own in the single-bunch, batched and
collective paths, at sizes below and above the one where a thread takes two particles.  Tolerance:
1e-10 of the bucket and of the transverse amplitude, the one of the maps' parity tests."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1610_05801_gb300 import phtl  # noqa: E402
from test_parity_gpu import run_ref  # noqa: E402
from test_widened_gpu import TOL, errors, widened_inputs  # noqa: E402

DEV = "cuda:0"
DUAL = dict(harmonic2=9240, voltage2_V=0.3 * 4.5e6, phi2_rad=0.0)
WIDE = dict(eta1=0.05, eta2=2.0, xi_x=5.0, xi_y=-3.0)
RINGS = {
    "zero": {}, "general": dict(phi_s=0.2), "linear": dict(rf_linear=1),
    "wide_zero": WIDE, "wide_general": dict(WIDE, phi_s=0.2), "wide_linear": dict(WIDE, rf_linear=1),
    "dual_plain": DUAL, "dual_phased": dict(DUAL, phi2_rad=-0.4), "dual_wide": dict(DUAL, **WIDE),
    "dual_general": dict(DUAL, phi_s=0.2, phi2_rad=0.3), "dual_linear": dict(DUAL, rf_linear=1),
}
TURNS = 200


def _run(inp, path, scheme):
    bufs = [torch.tensor(inp[k], dtype=torch.float64, device=DEV) for k in ("z", "dp", "x", "xp", "y", "yp")]
    R = phtl.Ring(**inp["ring"])
    if path == "batch":
        mon = torch.zeros(TURNS + 1, phtl.MON_FIELDS, dtype=torch.float64, device=DEV)
        B = phtl.Batch(R, [phtl.make_job(*bufs, turns=TURNS, integrator=scheme, dtype="f64", monitor=mon)])
        B.run()
        torch.cuda.synchronize()
        B.close()
    elif path == "collective":
        R.set_wake(np.zeros(16), -0.75, 0.75, 0.0)
        R.track_collective(*bufs, turns=TURNS, integrator=scheme)
    else:
        R.track(*bufs, turns=TURNS, integrator=scheme)
    torch.cuda.synchronize()
    R.close()
    return [b.cpu().numpy() for b in bufs]


@pytest.mark.parametrize("scheme", ["euler_cromer", "leapfrog", "ruth4", "rk4"])
@pytest.mark.parametrize("ring", sorted(RINGS))
def test_every_path_follows_the_oracle(ring, scheme):
    inp = widened_inputs(997, seed=7, **RINGS[ring])
    for k in ("z", "dp"):
        inp[k] = inp[k] * 0.4
    ref, _ = run_ref(inp, scheme, TURNS)
    for path in ("track", "batch", "collective"):
        err = errors(inp, _run(inp, path, scheme), ref)
        assert err < TOL["f64"][0], (path, err)


@pytest.mark.parametrize("ring", ["zero", "general", "linear"])
@pytest.mark.parametrize("scheme", ["leapfrog", "ruth4"])
def test_two_particles_a_thread(ring, scheme):
    inp = widened_inputs(40_001, seed=9, **RINGS[ring])
    for k in ("z", "dp"):
        inp[k] = inp[k] * 0.4
    ref, _ = run_ref(inp, scheme, TURNS)
    err = errors(inp, _run(inp, "track", scheme), ref)
    assert err < TOL["f64"][0], err
