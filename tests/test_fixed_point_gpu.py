"""The FP64 kernels' integer sines and integer moment sums at the edges of their ranges.

Sines: a kick of one Euler-Cromer turn from delta = 0 is kw * (sin(phi_s + k z) - sin(phi_s)),
so delta / kw after it is the device's sine to one rounding of each operation; the phases cover
the quarter-turn and half-turn borders, the borders of the integer form (a turn of k z), phases
of 1e-300 and zero, for phi_s = 0 and phi_s != 0.  Bound: 2 units of 2^-53 for the sine, one for each of the product and the
subtraction, and the phase's own rounding where it is formed in FP64.

Moments: raw sums of values of very different magnitude, signs and exact zeros against exact
rational sums; each warp's sums keep 2^-48 of its largest term (57-bit integers, products
2^-54), the additions of warps and blocks 2^-53 each.
"""
from fractions import Fraction
import math

import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from paper_1610_05801_gb300 import phtl, synth  # noqa: E402

DEV = "cuda:0"


def _longdouble_sin_minus(k, z, phi):
    x = np.longdouble(k) * z.astype(np.longdouble) + np.longdouble(phi)
    return np.sin(x) - np.sin(np.longdouble(phi))


@pytest.mark.parametrize("phi_s", [0.0, 0.3, -0.2])
def test_kick_sine_at_the_borders_of_its_forms(phi_s):
    ring = dict(synth.ring(4.5e6, transverse=False), phi_s_rad=phi_s)
    d = oracle.load().derive(ring)
    k = d.k
    turns = np.array([1 / 8, 1 / 4, 1 / 2, 3 / 4, 1.0, 1.5, 2.0, 3.25])
    z = [0.0, -0.0, 1e-300, -1e-300, 1e-12, -1e-12]
    for t in turns:
        c = t * 2 * math.pi / k
        for s in (1.0, -1.0):
            z += [s * c, s * np.nextafter(c, 0), s * np.nextafter(c, 9), s * c * (1 - 1e-10), s * c * (1 + 1e-10)]
    e = np.ldexp(1.0, np.arange(-40, 4))          # powers of two: every shift of the phase
    z = np.concatenate([np.array(z), e, -e, np.random.default_rng(0).uniform(-1.6, 1.6, 4001)])
    R = phtl.Ring(**ring)
    bz = torch.tensor(z, dtype=torch.float64, device=DEV)
    bd = torch.zeros_like(bz)
    R.track(bz, bd, turns=1, integrator="euler_cromer")
    got = bd.cpu().numpy()
    R.close()
    want = _longdouble_sin_minus(k, z, phi_s) * np.longdouble(d.A)
    # beyond the integer form the phase k z + phi_s is rounded to FP64: half a unit of its value
    tol = float(d.A) * 2.0 ** -53 * (4 + np.abs(k * z) + abs(phi_s))
    assert np.all(np.abs(got - want.astype(np.float64)) <= tol + np.spacing(np.abs(got)))
    if phi_s == 0.0:
        assert np.all(got[z == 0.0] == 0.0)
        tiny = (np.abs(k * z) < 1e-3) & (z != 0.0)
        assert np.max(np.abs(got[tiny] / want[tiny].astype(np.float64) - 1)) < 4e-16


@pytest.mark.parametrize("n", [1, 2, 31, 64, 65, 997])
@pytest.mark.parametrize("planes", [0, 2])
def test_moment_sums_of_mixed_magnitudes(n, planes):
    rng = np.random.default_rng(n)
    coords = []
    for i in range(2 + 2 * planes):
        a = rng.normal(0, 1, n) * 10.0 ** rng.integers(-9, 3, n) * 10.0 ** (-3 * i)
        a[rng.random(n) < 0.2] = 0.0
        coords.append(a)
    coords[0][-1] = 1e-300          # shifted out next to the others, exact alone
    bufs = [torch.tensor(a, dtype=torch.float64, device=DEV) for a in coords]
    bufs += [None] * (6 - len(bufs))
    mon = torch.zeros(1, phtl.MON_FIELDS, dtype=torch.float64, device=DEV)
    R = phtl.Ring(**synth.ring(4.5e6, transverse=True))
    R.set_monitor(mon, stride=1)
    R.track(*bufs, turns=0)
    row = mon.cpu().numpy()[0]
    R.close()
    assert row[0] == n
    for plane in range(1 + planes):
        a, b = ([Fraction(float(v)) for v in coords[2 * plane + j]] for j in (0, 1))
        ma, mb = max(map(abs, a)), max(map(abs, b))
        tol = 2.0 ** -47 + n * 2.0 ** -53
        for j, (u, v, big) in enumerate(((a, None, ma), (b, None, mb), (a, a, ma * ma), (b, b, mb * mb),
                                         (a, b, ma * mb))):
            # the exact sum as FP64 holds it (1e-300 squared is zero there)
            exact = Fraction(float(sum(u) if v is None else sum(p * q for p, q in zip(u, v))))
            assert abs(Fraction(float(row[1 + 5 * plane + j])) - exact) <= Fraction(tol) * big * max(1, n // 64 + 1), (plane, j)
    assert np.all(row[1 + 5 * (1 + planes):] == 0)


def test_moments_of_non_finite_values_are_nan():
    z = np.array([0.1, np.inf, -0.2, 0.3])
    dp = np.array([1e-3, 2e-3, -1e-3, 0.0])
    bufs = [torch.tensor(a, dtype=torch.float64, device=DEV) for a in (z, dp)]
    mon = torch.zeros(1, phtl.MON_FIELDS, dtype=torch.float64, device=DEV)
    R = phtl.Ring(**synth.ring(4.5e6, transverse=False))
    R.set_monitor(mon, stride=1)
    R.track(*bufs, turns=0)
    row = mon.cpu().numpy()[0]
    R.close()
    assert row[0] == 4 and np.all(np.isnan(row[[1, 3, 5]]))
    assert abs(row[2] - 2e-3) < 1e-18 and abs(row[4] - 6e-6) < 1e-20


@pytest.mark.parametrize("planes, small, large", [(0, 4097, 240_001), (2, 4097, 60_001)])
@pytest.mark.parametrize("stride", [0, 1])
def test_small_bunches_track_as_inside_large_ones(planes, small, large, stride):
    """Bunches below and above the size at which a thread takes two particles instead of one: the
    same particles bitwise, and moments of the small bunch against its own coordinates' sums."""
    ring = synth.ring(4.5e6, transverse=True)
    rng = np.random.default_rng(7)
    coords = [rng.normal(0, 0.15, large), rng.normal(0, 1e-3, large)]
    for _ in range(planes):
        coords += [rng.normal(0, 2e-3, large), rng.normal(0, 4e-5, large)]
    out = []
    for n in (small, large):
        R = phtl.Ring(**ring)
        bufs = [torch.tensor(a[:n], dtype=torch.float64, device=DEV) for a in coords]
        mon = torch.zeros(26, phtl.MON_FIELDS, dtype=torch.float64, device=DEV)
        if stride:
            R.set_monitor(mon, stride=stride)
        R.track(*bufs, *[None] * (6 - len(bufs)), turns=25, integrator="leapfrog")
        out.append([b[:small].cpu().numpy() for b in bufs])
        if stride and n == small:
            row, a = mon.cpu().numpy()[25], out[0]
            assert row[0] == n
            for i in range(1 + planes):
                u, v = a[2 * i], a[2 * i + 1]
                want = [u.sum(), v.sum(), u @ u, v @ v, u @ v]
                scale = [np.abs(u).sum(), np.abs(v).sum(), u @ u, v @ v, np.abs(u) @ np.abs(v)]
                assert np.all(np.abs(row[1 + 5 * i:6 + 5 * i] - want) <= 1e-12 * np.array(scale))
        R.close()
    for u, v in zip(*out):
        assert np.array_equal(u, v)


@pytest.mark.parametrize("k", [2 * math.pi * 4620 / 6911.5, 1.0, 0.037])
def test_sine_of_a_negative_wave_number(k):
    """sin(-k z) = -sin(k z) bitwise, and within 2 units of 2^-53 of the exact sine, in the bucket, some
    turns and many turns away."""
    rng = np.random.default_rng(3)
    ph = np.concatenate([rng.uniform(-3, 3, 3001), rng.uniform(-60, 60, 3001), rng.uniform(-9e4, 9e4, 3001)])
    z = torch.tensor(ph / k, dtype=torch.float64, device=DEV)
    a, b = phtl.eval_sin_kz(k, z).cpu().numpy(), phtl.eval_sin_kz(-k, z).cpu().numpy()
    assert np.array_equal(a, -b)
    want = _longdouble_sin_minus(k, z.cpu().numpy(), 0.0)
    # the reference's own phase, in the host's long double (64 bits at least): half a unit of it
    tol = 2 * 2.0 ** -53 + np.abs(ph) * float(np.finfo(np.longdouble).eps)
    assert np.all(np.abs((a - want).astype(np.float64)) <= tol)
