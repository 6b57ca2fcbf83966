"""PHTL_F32C forms the RF phase in FP64: kicks at small phases, where the phase's rounding is not
covered by the sine polynomial's error.

One Euler-Cromer turn from delta = 0 leaves delta = A sin(k z) as a float pair.  The operations of that
kick, evaluated one by one on the host for 3e5 particles between 1 um and 1 mm, leave a relative error of
0.73 2^-48 rms with the phase in FP64 (split to 2^-48) and of 0.92 2^-48 with a phase formed from the
coordinate's floats; 0.70 with every product renormalised.  Bound: 0.8 2^-48, the middle, for the rms of
2e5 particles (its own scatter is below 0.01), and 8 2^-48 for each.
"""
import math

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1610_05801_gb300 import phtl, synth  # noqa: E402

DEV = "cuda:0"
UNIT = 2.0 ** -48


@pytest.mark.parametrize("path", ["track", "perturn", "batch", "collective"])
def test_small_phase_kicks(path):
    n = 200_001
    rng = np.random.default_rng(3)
    z = phtl.split_f32c(10.0 ** rng.uniform(-6, -3, n) * rng.choice([-1.0, 1.0], n))
    ring = synth.ring(4.5e6, transverse=False)
    d = oracle.load().derive(ring)
    R = phtl.Ring(**ring)
    bz = torch.tensor(z, dtype=torch.float32, device=DEV)
    bd = torch.zeros_like(bz)
    opt = dict(turns=1, integrator="euler_cromer", dtype="f32c")
    if path == "batch":
        B = phtl.Batch(R, [phtl.make_job(bz, bd, **opt)])
        B.run()
        torch.cuda.synchronize()
        B.close()
    elif path == "collective":
        R.set_wake(np.zeros(16), -0.75, 0.75, 0.0)
        R.track_collective(bz, bd, **opt)
    else:
        (R.track if path == "track" else R.track_perturn)(bz, bd, **opt)
    torch.cuda.synchronize()
    R.close()
    x = np.longdouble(d.k) * phtl.join_f32c(z).astype(np.longdouble)
    want = np.longdouble(d.A) * np.sin(x)
    pair = bd.cpu().numpy()
    got = pair[:n].astype(np.longdouble) + pair[n:].astype(np.longdouble)
    rel = ((got - want) / want).astype(np.float64) / UNIT
    assert math.sqrt(float(np.mean(rel * rel))) <= 0.8
    assert float(np.max(np.abs(rel))) <= 8.0


def test_tails_of_coordinates_whose_head_is_zero():
    """Coordinates as a caller may hand them over, not normalised: hi = 0 and a compensation from 1e-36 to
    1e-9, beside exact zeros.  sin(k z) is k z there, to the pairs' 8 2^-48 and FP32's smallest normal number."""
    comp = np.concatenate([[0.0, -0.0], np.logspace(-36, -9, 28), -np.logspace(-36, -9, 28)]).astype(np.float32)
    n = comp.size
    d = oracle.load().derive(synth.ring(4.5e6, transverse=False))
    R = phtl.Ring(**synth.ring(4.5e6, transverse=False))
    bz = torch.tensor(np.concatenate([np.zeros(n, dtype=np.float32), comp]), device=DEV)
    bd = torch.zeros_like(bz)
    R.track(bz, bd, turns=1, integrator="euler_cromer", dtype="f32c")
    torch.cuda.synchronize()
    R.close()
    got = phtl.join_f32c(bd.cpu().numpy())
    want = d.A * d.k * comp.astype(np.float64)
    assert np.all(np.abs(got - want) <= 8 * UNIT * np.abs(want) + 2.0 ** -126 * 1e-3)
    assert np.all(got[:2] == 0.0)
