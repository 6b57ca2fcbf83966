"""FP64 kicks at small phases: a kick is exact relative to its own terms, not only to 1.

One turn from delta = 0 with |z| between 1 nm and 1 mm, against the map in the host's long double.
The sine of a small phase has the phase's relative precision, so each term of the kick carries a few
units of 2^-53 of max(|sin(phi + k z)|, |sin phi|): 1.1 for the sine, 1.5 for sin phi and the
subtraction, 1 for the stage's weight, 2 for the multiply-adds of the term and of the sum, 1 more for
RK4's weighted sum; 8 in all, over the sum of the stages' terms.  A phase kept to a fixed fraction of a
turn instead misses this by up to 1e8 at 1 nm.
"""
import math

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1610_05801_gb300 import phtl, synth  # noqa: E402

DEV = "cuda:0"
LD = np.longdouble
UNITS = 8 * 2.0 ** -53
THETA = LD(1) / (LD(2) - LD(2) ** (LD(1) / LD(3)))
STAGES = {"euler_cromer": (("k", LD(1)), ("d", LD(1))),
          "leapfrog": (("d", LD(0.5)), ("k", LD(1)), ("d", LD(0.5))),
          "ruth4": (("d", THETA / 2), ("k", THETA), ("d", (1 - THETA) / 2), ("k", 1 - 2 * THETA),
                    ("d", (1 - THETA) / 2), ("k", THETA), ("d", THETA / 2))}


def _z():
    rng = np.random.default_rng(11)
    a = 10.0 ** rng.uniform(-9, -3, 3001)
    return np.concatenate([a, -a, [0.0]])


def _one_turn(systems, etaC, e1C, e2C, scheme, z0):
    """(delta, bound) after one turn from delta = 0; systems: (A, k, phi) of each RF system."""
    z, d, scale = z0.astype(LD), np.zeros_like(z0, dtype=LD), np.zeros_like(z0, dtype=LD)

    def force(z):
        f, s = LD(0), LD(0)
        for A, k, phi in systems:
            a, b = np.sin(LD(phi) + LD(k) * z), np.sin(LD(phi))
            f = f + LD(A) * (a - b)
            s = s + abs(A) * np.maximum(np.abs(a), np.abs(b))
        return f, s

    def slip(d):
        return ((LD(e2C) * d + LD(e1C)) * d + LD(etaC)) * d

    if scheme == "rk4":
        a1, (b1, s1) = -slip(d), force(z)
        a2, (b2, s2) = -slip(d + b1 / 2), force(z + a1 / 2)
        a3, (b3, s3) = -slip(d + b2 / 2), force(z + a2 / 2)
        b4, s4 = force(z + a3)
        return d + (b1 + 2 * b2 + 2 * b3 + b4) / 6, (s1 + 2 * s2 + 2 * s3 + s4) / 6
    for what, w in STAGES[scheme]:
        if what == "k":
            f, s = force(z)
            d, scale = d + w * f, scale + abs(w) * s
        else:
            z = z - w * slip(d)
    return d, scale


def _check(got, want, scale):
    err = np.abs((got.astype(LD) - want).astype(np.float64))
    worst = float(np.max(err / np.maximum(UNITS * scale.astype(np.float64), 1e-300)))
    assert worst <= 1.0, worst


def _run(ring, scheme, programme=None):
    z = _z()
    R = phtl.Ring(**ring)
    bz = torch.tensor(z, dtype=torch.float64, device=DEV)
    bd = torch.zeros_like(bz)
    if programme:
        R.set_programme(*programme)
        R.track_programme(bz, bd, turn0=0, turns=1, integrator=scheme)
    else:
        R.track(bz, bd, turns=1, integrator=scheme)
    torch.cuda.synchronize()
    R.close()
    return z, bd.cpu().numpy()


@pytest.mark.parametrize("scheme", ["euler_cromer", "leapfrog", "ruth4", "rk4"])
@pytest.mark.parametrize("phi2", [0.0, 1e-9, -1e-3])
@pytest.mark.parametrize("ratio", [0.3, -0.5])
@pytest.mark.parametrize("slippage", [False, True])
def test_second_rf_system(scheme, phi2, ratio, slippage):
    ring = dict(synth.ring(4.5e6, transverse=False), harmonic2=9240, voltage2_V=ratio * 4.5e6, phi2_rad=phi2)
    if slippage:
        ring.update(eta1=0.05, eta2=2.0)
    d = oracle.load().derive(ring)
    z, got = _run(ring, scheme)
    _check(got, *_one_turn(((d.A, d.k, 0.0), (d.A2, d.k2, phi2)), d.etaC, d.eta1C, d.eta2C, scheme, z))


@pytest.mark.parametrize("scheme", ["euler_cromer", "leapfrog", "ruth4", "rk4"])
@pytest.mark.parametrize("phi_s", [1e-9, -1e-6, 1e-3])
def test_small_synchronous_phase(scheme, phi_s):
    ring = dict(synth.ring(4.5e6, transverse=False), phi_s_rad=phi_s)
    d = oracle.load().derive(ring)
    z, got = _run(ring, scheme)
    _check(got, *_one_turn(((d.A, d.k, phi_s),), d.etaC, 0.0, 0.0, scheme, z))


@pytest.mark.parametrize("scheme", ["euler_cromer", "leapfrog", "ruth4"])
@pytest.mark.parametrize("gain", [0.0, 4.5e-3, 4.5e3])
def test_programme_at_and_near_constant_momentum(scheme, gain):
    """Momentum gains of 0, 4.5 meV/c and 4.5 keV/c a turn: phi_s,n of 0, 1e-9 and 1e-3."""
    ring = synth.ring(4.5e6, transverse=False)
    d = oracle.load().derive(ring)
    p0 = np.array([26e9, 26e9 + gain])
    z, got = _run(ring, scheme, (np.array([4.5e6]), p0))
    bg = p0[0] / 938.27208816e6
    phis = math.asin(bg / math.sqrt(1.0 + bg * bg) * (p0[1] - p0[0]) / 4.5e6)
    want, scale = _one_turn(((d.A, d.k, phis),), d.etaC, 0.0, 0.0, scheme, z)
    r = LD(p0[0]) / LD(p0[1])
    _check(got, want * r, scale)
