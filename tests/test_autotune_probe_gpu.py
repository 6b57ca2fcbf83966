"""The autotuner's probe runs what a batch runs: its rate on a double-RF ring is the batch's.

The probe is one launch that fills the GPU once, a batch several with a fuller last round, so the probe's
rate is 0.7 to 0.95 of a batch's on every ring; particles that the kicks answer out of line (the centre of
the second RF system, once) halve it.  Bound: 0.65 of the measured batch, best of five runs.
"""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1610_05801_gb300 import phtl, synth  # noqa: E402

DEV = "cuda:0"
N, TURNS = 2_000_001, 100


@pytest.mark.parametrize("scheme", ["leapfrog", "ruth4"])
def test_probe_rate_on_a_double_rf_ring(scheme):
    R = phtl.Ring(**synth.ring(4.5e6, transverse=False, harmonic2=9240, voltage2_V=0.3 * 4.5e6))
    gen = torch.Generator(device=DEV)
    gen.manual_seed(1)
    z = 0.15 * torch.randn(N, generator=gen, device=DEV, dtype=torch.float64)
    dp = 1e-3 * torch.randn(N, generator=gen, device=DEV, dtype=torch.float64)
    rate = R.autotune("f64", scheme, active_particles=N).particle_turns_per_s
    B = phtl.Batch(R, [phtl.make_job(z, dp, turns=TURNS, integrator=scheme, dtype="f64")])
    best = float("inf")
    for i in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        B.run()
        e1.record()
        torch.cuda.synchronize()
        if i:
            best = min(best, e0.elapsed_time(e1))
    B.close()
    R.close()
    assert rate > 0.65 * N * TURNS / (best * 1e-3), (rate, N * TURNS / (best * 1e-3))
