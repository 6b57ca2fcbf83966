"""The FP64 kernels' integer sines, chromatic phases and moment sums within the bounds that their forms
have, derived here term by term (test_fixed_point_gpu.py checks the same forms within wider ones).

u is 2^-53, the relative bound of one rounding.

Kicks (Euler-Cromer from delta = 0): the fixed-point sine is within 0.75 u of the exact one at any number
of turns (half a unit of its rounding below 1, the cuts of phase and polynomial at 2^-60); a phase adds
0.5 u for the rounded sin(phi) and u |f| for the subtraction; the kick's multiply-adds of up to two
systems round f's product and the sum: 2 u |f|.

Chromatic plane: the device's sine times beta and sine over beta are within 1 u of beta and of 1/beta
(0.75, and half a unit of 1/beta), the cosine within 0.75 u; each output is a product and a multiply-add:
u of the product and of the sum.  From half a turn of xi delta on, and where the sine does not fill the
significand (below 2^-24), the phase may be the FP64 fma(xi, delta, q), u of its value times 2 pi, with
one rounding more.

Moments: a thread's sum of values is cut once below 2^-56 of the warp's largest, 32 lanes: 2^-51, and the
values themselves below 2^-60, 64 of them; of products below 2^-55, up to 2.5 units each, 32 lanes:
2^-48.6; then one rounding per warp and one per addition of a warp's total.
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
LD = np.longdouble
EPS_LD = float(np.finfo(LD).eps)


def _kick_positions(k):
    rng = np.random.default_rng(2)
    z = [rng.uniform(-1, 1, 4001) * t * 2 * math.pi / k for t in (0.5, 1.0, 2.0, 8.0, 100.0, 1.4e4)]
    for turns in (1 / 8, 1 / 4, 1 / 2, 3 / 4, 1.0, 1.5, 2.0, 8.0, 16.0, 1000.0):
        c = turns * 2 * math.pi / k
        z.append(np.array([s * v for s in (1, -1) for v in (c, np.nextafter(c, 0), np.nextafter(c, 1e9),
                                                            c * (1 - 1e-10), c * (1 + 1e-10), c * (1 - 1e-6))]))
    return np.concatenate(z)


@pytest.mark.parametrize("phi_s", [0.0, 0.3, -0.2, 1.2])
@pytest.mark.parametrize("second", [None, 0.0, 0.7])
def test_kicks(phi_s, second):
    over = {} if second is None else dict(harmonic2=9240, voltage2_V=1.35e6, phi2_rad=second)
    ring = dict(synth.ring(4.5e6, transverse=False, **over), phi_s_rad=phi_s)
    d = oracle.load().derive(ring)
    z = _kick_positions(d.k)
    if second is not None:  # both systems' phases below 1e5 radians
        z = z[np.abs(z * d.k2) < 9e4]
    R = phtl.Ring(**ring)
    bz = torch.tensor(z, dtype=torch.float64, device=DEV)
    bd = torch.zeros_like(bz)
    R.track(bz, bd, turns=1, integrator="euler_cromer")
    got = bd.cpu().numpy().astype(LD)
    R.close()
    want, tol = np.zeros(z.size, dtype=LD), np.zeros(z.size)
    for A, k, phi in ((d.A, d.k, phi_s),) + (() if second is None else ((d.A2, d.k2, second),)):
        x = LD(k) * z.astype(LD) + LD(phi)
        f = np.sin(x) - np.sin(LD(phi))
        want = want + LD(A) * f
        f = np.abs(f.astype(np.float64))
        units = 0.75 + (0.5 + f if phi else 0.0) + 2.0 * f
        tol += abs(A) * (units * 2.0 ** -53 + (np.abs(k * z) + 2) * EPS_LD)
    err = np.abs((got - want).astype(np.float64))
    assert np.all(err <= tol), float(np.max(err / tol))


@pytest.mark.parametrize("xi", [5.0, -3.0, 0.25])
@pytest.mark.parametrize("n", [1, 4001])
def test_chromatic_rotation_at_its_borders(xi, n):
    ring = synth.ring(4.5e6, transverse=True, xi_x=xi, xi_y=-xi)
    dv = oracle.load().derive(ring)
    rng = np.random.default_rng(4)
    delta = [0.0, -0.0, 1e-300, -1e-300, 5e-324, 1e-12, -1e-12]
    for q in (dv.qx, dv.qy):
        for turns in (0.0, 1 / 4, 1 / 2, 3 / 4, 1.0, 1.5, 2.0, 5.0):  # of the whole phase, and of xi delta
            for c in ((turns - q) / xi, -(turns - q) / xi, turns / xi, -turns / xi):
                delta += [c, np.nextafter(c, 0), np.nextafter(c, 9 * np.sign(c)), c * (1 - 1e-10), c * (1 + 1e-10)]
    delta = np.concatenate([np.array(delta), rng.uniform(-1.5, 1.5, 4001) / abs(xi)])
    if n == 1:
        delta = delta[60:61]
    m = delta.size
    u, v = rng.normal(0, 2e-3, (2, m)), rng.normal(0, 4e-5, (2, m))
    R = phtl.Ring(**ring)
    bufs = [torch.tensor(a, dtype=torch.float64, device=DEV)
            for a in (np.zeros(m), delta, u[0], v[0], u[1], v[1])]
    R.track(*bufs, turns=1, integrator="euler_cromer")  # z = 0: the kick is zero
    got = [b.cpu().numpy() for b in bufs]
    R.close()
    assert np.array_equal(got[1], delta)
    for p, (q, b) in enumerate(((dv.qx, dv.bx), (dv.qy, dv.by))):
        s = xi if p == 0 else -xi
        a = LD(q) + LD(s) * delta.astype(LD)
        mu = 2 * LD("3.14159265358979323846264338327950288") * (a - np.rint(a))
        cs, sn = np.cos(mu), np.sin(mu)
        wide = (np.abs(s * delta) >= 0.5) | (np.abs(sn) < 2.0 ** -24)
        phase = np.where(wide, 2 * math.pi * np.abs(a.astype(np.float64)) + 2.0, 0.0)
        ua, va = np.abs(u[p]), np.abs(v[p])
        c, n_ = np.abs(cs).astype(np.float64), np.abs(sn).astype(np.float64)
        for g, want, x, y in ((got[2 + 2 * p], cs * u[p].astype(LD) + LD(b) * sn * v[p].astype(LD), ua, b * va),
                              (got[3 + 2 * p], cs * v[p].astype(LD) - sn / LD(b) * u[p].astype(LD), va, ua / b)):
            tol = 2.0 ** -53 * (y + 0.75 * x + 2.0 * c * x + n_ * y + (x + y) * phase) + (x + y) * 16 * EPS_LD
            err = np.abs((g.astype(LD) - want).astype(np.float64))
            assert np.all(err <= tol), (p, float(np.max(err / tol)))


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 64, 65, 997, 70_001])
@pytest.mark.parametrize("planes", [0, 2])
def test_moment_sums(n, planes):
    rng = np.random.default_rng(n)
    coords = []
    for i in range(2 + 2 * planes):
        a = rng.normal(0, 1, n) * 10.0 ** rng.integers(-9, 3, n) * 10.0 ** (-3 * i)
        a[rng.random(n) < 0.2] = 0.0
        coords.append(a)
    bufs = [torch.tensor(a, dtype=torch.float64, device=DEV) for a in coords] + [None] * (4 - 2 * planes)
    mon = torch.zeros(1, phtl.MON_FIELDS, dtype=torch.float64, device=DEV)
    R = phtl.Ring(**synth.ring(4.5e6, transverse=True))
    R.set_monitor(mon, stride=1)
    R.track(*bufs, turns=0)
    row = mon.cpu().numpy()[0]
    R.close()
    assert row[0] == n
    warps = -(-n // 32)
    for plane in range(1 + planes):
        a, b = coords[2 * plane], coords[2 * plane + 1]
        ma, mb = float(np.max(np.abs(a))), float(np.max(np.abs(b)))
        fa, fb = ([Fraction(float(v)) for v in c] for c in (a, b))
        for j, (terms, cut) in enumerate(((fa, 2.0 ** -50.9 * ma), (fb, 2.0 ** -50.9 * mb),
                                          ([v * v for v in fa], 2.0 ** -48.6 * ma * ma),
                                          ([v * v for v in fb], 2.0 ** -48.6 * mb * mb),
                                          ([v * w for v, w in zip(fa, fb)], 2.0 ** -48.6 * ma * mb))):
            exact, total = sum(terms), float(sum(map(abs, terms)))
            tol = warps * cut + (warps + 1) * 2.0 ** -53 * total
            assert abs(Fraction(float(row[1 + 5 * plane + j])) - exact) <= Fraction(tol), (plane, j)
