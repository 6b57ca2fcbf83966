"""Timed cases of the tracker: what its users have it do, through the public entry points.

listed() gives the cases, draw() more of the same families and ranges, prepare() what a
program holds before the call (seeded inputs on the GPU, the ring handle, a batch), run()
one pass as a program makes it, work() the bytes and operations a pass cannot do without and
exact() its results from plain torch in 64 bits.

The ring is the one of the benchmark (C = 6911.5 m, h = 4620, p0 = 26 GeV/c, gamma_t = 22.77);
bunches are matched Gaussians (sigma_z = 0.15 m) inside 95 % of the separatrix, or the
core-and-halo bunch of the precision sweep, with Gaussian transverse planes.  The sizes are the
benchmark's with fewer turns per pass; a program calls track() again and again on the same
particles, and so does a repeated run().
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1610_05801_gb300 import phtl

MASS = 938.27208816e6
RING = dict(circumference_m=6911.5, harmonic=4620, p0_eVc=26e9, gamma_t=22.77, mass_eV=MASS,
            charge_e=1.0, phi_s_rad=0.0, beta_x_m=50.0, beta_y_m=50.0, Qx=20.13, Qy=20.18)
WIDENED = dict(eta1=0.05, eta2=2.0, xi_x=5.0, xi_y=-3.0)
DUAL = dict(harmonic2=9240, voltage2_V=0.3 * 4.5e6, phi2_rad=0.0)
VOLTAGE = 4.5e6
SCHEMES = ("euler_cromer", "leapfrog", "ruth4")
DTYPES = ("f64", "f32c", "f32cd", "f32cs")
WAKE_LO, WAKE_HI, WAKE_ALPHA, WAKE_SC = -0.75, 0.75, -5e-11, 1e-9


# ---- the cases -------------------------------------------------------------------------

def listed():
    return [
        # the smallest job: 1000 particles for 1000 turns, longitudinal only; latency
        dict(name="small_f64", kind="track", n=1000, turns=1000, scheme="leapfrog", dtype="f64",
             planes=0, stride=0, map="linear", halo=False),
        # the paper-scale single bunch: the three schemes one after another on a million
        # particles with both transverse planes, moments after every turn
        dict(name="paper_f64", kind="schemes", n=1_000_000, turns=300, dtype="f64", planes=2, stride=1),
        # a ragged bunch without turn-by-turn moments, one transverse plane, 4th order
        dict(name="ragged_ruth4_f64", kind="track", n=300_007, turns=500, scheme="ruth4", dtype="f64",
             planes=1, stride=0, map="linear", halo=False),
        # the precision sweep's bunch: four million particles, core and halo, longitudinal,
        # FP32-compensated arithmetic with the phase formed in FP64
        dict(name="halo_f32c", kind="track", n=4_000_000, turns=200, scheme="leapfrog", dtype="f32c",
             planes=0, stride=0, map="linear", halo=True),
        # FP32-compensated without FP64 instructions, transverse planes and moments, odd size
        dict(name="ruth4_f32cd", kind="track", n=250_001, turns=400, scheme="ruth4", dtype="f32cd",
             planes=2, stride=1, map="linear", halo=False),
        # uneven bunches of different voltage and length in one graph-captured batch with
        # moments after every turn, FP32-compensated
        dict(name="batch_f32c", kind="batch", bunches=64, total=6_000_000, turns_lo=50, turns_hi=1000,
             mix=False, seed0=3),
        # what the serving loop hands to the batched kernels: schemes and arithmetic mixed
        dict(name="batch_mixed", kind="batch", bunches=24, total=3_000_000, turns_lo=50, turns_hi=500,
             mix=True, seed0=4),
        # nonlinear slippage and chromaticity, moments every 10 turns
        dict(name="widened_lf_f64", kind="track", n=1_000_000, turns=100, scheme="leapfrog",
             dtype="f64", planes=2, stride=10, map="widened", halo=False),
        # classic Runge-Kutta on a double-RF ring
        dict(name="rk4_dual_f64", kind="track", n=500_000, turns=100, scheme="rk4", dtype="f64",
             planes=2, stride=1, map="dual", halo=False),
        # an accelerating bucket: voltage and momentum programme
        dict(name="ramp_lf_f64", kind="ramp", n=500_000, turns=300, scheme="leapfrog", dtype="f64",
             planes=2, stride=1),
        # slicing, wake and space-charge kick after every turn
        dict(name="collective_lf_f64", kind="collective", n=1_000_000, turns=100, scheme="leapfrog",
             dtype="f64", planes=2, stride=10, slices=512),
        # the call on host buffers: copies in and out, moments back
        dict(name="host_lf_f64", kind="host", n=100_000, turns=300, scheme="leapfrog", dtype="f64",
             planes=2, stride=10),
    ]


def _loguniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


_FLOP_CAP = 3e10  # below the paper-scale case


def _fit(rng, case):
    """Turns for the case's particles: log-uniform, within the largest listed case's work."""
    per = _flops_per_turn(case)
    hi = max(20, min(1500, int(_FLOP_CAP / (per * case["n"]))))
    case["turns"] = _loguniform(rng, 20, hi) if hi > 20 else 20
    return case


def draw(rng):
    kind = rng.choice(("track", "track", "track", "track", "batch", "widened", "dual", "ramp",
                       "collective", "host"))
    n = _loguniform(rng, 500, 3_000_000) | rng.randint(0, 1)
    dtype = rng.choice(("f64", "f64", "f32c", "f32cd", "f32cs"))
    planes, stride = rng.choice((0, 1, 2, 2)), rng.choice((0, 1, 1, 10))
    scheme = rng.choice(SCHEMES)
    if kind == "batch":
        lo = rng.randint(20, 100)
        return dict(kind="batch", bunches=rng.randint(4, 64), total=_loguniform(rng, 100_000, 4_000_000),
                    turns_lo=lo, turns_hi=lo * rng.randint(2, 8), mix=rng.random() < 0.5,
                    seed0=rng.randint(10, 1 << 20))
    if kind in ("widened", "dual"):
        return _fit(rng, dict(kind="track", n=min(n, 1_000_001), turns=0, dtype=dtype, planes=planes,
                              stride=stride, scheme=rng.choice(SCHEMES + ("rk4",)), map=kind, halo=False))
    if kind == "ramp":
        return _fit(rng, dict(kind="ramp", n=n, turns=0, scheme=scheme, dtype=dtype, planes=planes,
                              stride=stride))
    if kind == "collective":
        return _fit(rng, dict(kind="collective", n=n, turns=0, scheme=scheme, dtype=dtype,
                              planes=planes, stride=stride, slices=rng.choice((64, 200, 512, 1000))))
    if kind == "host":
        return _fit(rng, dict(kind="host", n=min(n, 1_000_001), turns=0, scheme=scheme, dtype=dtype,
                              planes=planes, stride=stride))
    return _fit(rng, dict(kind="track", n=n, turns=0, scheme=scheme, dtype=dtype, planes=planes,
                          stride=stride, map="linear", halo=rng.random() < 0.3))


# ---- inputs ----------------------------------------------------------------------------

def _ring(case):
    r = dict(RING, voltage_V=VOLTAGE)
    if case.get("map") == "widened":
        r.update(WIDENED)
    if case.get("map") == "dual":
        r.update(DUAL)
    return r


def _consts(r, p0=None, voltage=None):
    """(k, A, eta C, beta gamma) of a ring."""
    p0 = r["p0_eVc"] if p0 is None else p0
    bg = p0 / r["mass_eV"]
    g = math.sqrt(1.0 + bg * bg)
    eta = 1.0 / (r["gamma_t"] * r["gamma_t"]) - 1.0 / (g * g)
    k = 2.0 * math.pi * r["harmonic"] / r["circumference_m"]
    A = r["charge_e"] * (r["voltage_V"] if voltage is None else voltage) / ((bg / g) * p0)
    return k, A, eta * r["circumference_m"], bg


def _bunch(gen, n, planes, ring, voltage=VOLTAGE, halo=False, scale=1.0):
    """z, dp and up to two transverse planes of n particles, float64 on the GPU."""
    k, A, eC, bg = _consts(ring, voltage=voltage)
    zb, db = math.pi / k, 2.0 * math.sqrt(A / (k * eC))
    sz = 0.15
    sd = sz * math.sqrt(eC * A * k) / eC
    top = (A / k) * (1.0 - math.cos(0.95 * math.pi))

    def fill(m, one):
        got, have = [], 0
        while have < m:
            z, d = one(max(1024, int(1.5 * (m - have))))
            ok = 0.5 * eC * d * d + (A / k) * (1.0 - torch.cos(k * z)) <= top
            z, d = z[ok], d[ok]
            got.append((z, d))
            have += z.numel()
        return torch.cat([a for a, _ in got])[:m], torch.cat([b for _, b in got])[:m]

    def normal(m):
        return torch.randn(m, generator=gen, device="cuda", dtype=torch.float64)

    def uniform(m):
        return 2.0 * torch.rand(m, generator=gen, device="cuda", dtype=torch.float64) - 1.0

    core = n if not halo else int(round(0.6 * n))
    z, d = fill(core, lambda m: (normal(m) * sz, normal(m) * sd))
    if halo:
        zh, dh = fill(n - core, lambda m: (uniform(m) * zb, uniform(m) * db))
        at = torch.randperm(n, generator=gen, device="cuda")
        z, d = torch.cat([z, zh])[at], torch.cat([d, dh])[at]
    c = [z * scale, d * scale]
    eps = 2e-6 / bg
    for plane in range(2):
        if plane < planes:
            c += [normal(n) * math.sqrt(50.0 * eps), normal(n) * math.sqrt(eps / 50.0)]
        else:
            c += [None, None]
    return [None if a is None else a.contiguous() for a in c]


def _pack(a, dtype):
    """The library's layout of an arithmetic type: doubles, or [hi | comp] floats."""
    if a is None or dtype == "f64":
        return a
    hi = a.float()
    return torch.cat([hi, (a - hi.double()).float()])


def _unpack(b, dtype):
    if b is None or dtype == "f64":
        return b
    n = b.numel() // 2
    return b[:n].double() + b[n:].double()


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _rows(turns, stride):
    return torch.zeros(turns // stride + 1, phtl.MON_FIELDS, dtype=torch.float64, device="cuda")


def _batch_jobs(case):
    """Sizes, turns, voltages, schemes and types of the batch's bunches (host numbers)."""
    r = np.random.default_rng(case["seed0"])
    m = case["bunches"]
    n = np.exp(r.uniform(math.log(1e3), math.log(4e6), m))
    n = np.maximum((n * (case["total"] / n.sum())).astype(np.int64), 100) | 1
    jobs = []
    for i in range(m):
        jobs.append(dict(n=int(n[i]), turns=int(r.integers(case["turns_lo"], case["turns_hi"] + 1)),
                         voltage=float(r.uniform(1e6, 6e6)),
                         scheme=SCHEMES[int(r.integers(3))] if case["mix"] else "leapfrog",
                         dtype=("f64" if r.random() < 0.5 else "f32c") if case["mix"] else "f32c"))
    return jobs


def _slot(job):
    """Elements that one coordinate of a bunch takes in its batch's array."""
    per = job["n"] * (1 if job["dtype"] == "f64" else 2)
    return (per + 63) // 64 * 64


def _programme(case):
    """Voltage and momentum of the ramp: 2 MeV/c per turn from 26 GeV/c."""
    turns = case["turns"]
    return np.full(turns, VOLTAGE), RING["p0_eVc"] + 2e6 * np.arange(turns + 1, dtype=np.float64)


def _wake(case):
    m = np.arange(case["slices"], dtype=np.float64)
    return np.exp(-m / (case["slices"] / 10.0)) * np.cos(m / (case["slices"] / 20.0))


def _inputs(case, seed):
    """Initial coordinates in 64 bits, [planes] per bunch."""
    gen, kind = _gen(seed), case["kind"]
    if kind == "batch":
        return [_bunch(gen, j["n"], 0, dict(RING, voltage_V=VOLTAGE), voltage=j["voltage"])
                for j in _batch_jobs(case)]
    one = _bunch(gen, case["n"], case["planes"], _ring(case), halo=case.get("halo", False),
                 scale=0.3 if kind == "ramp" else 1.0)
    if kind == "schemes":
        return [[None if a is None else a.clone() for a in one] for _ in SCHEMES]
    return [one]


def prepare(case, seed):
    kind = case["kind"]
    state = dict(case=case, ring=phtl.Ring(**_ring(case)))
    R, start = state["ring"], _inputs(case, seed)
    if kind == "batch":
        # the bunches of a type lie one after another in one allocation, each 256-byte aligned
        plan = _batch_jobs(case)
        total, row = dict(f64=0, f32c=0), 0
        for j in plan:
            j["at"], j["row"] = total[j["dtype"]], row
            total[j["dtype"]] += 2 * _slot(j)
            row += j["turns"] + 1
        state["out"] = dict(f64=torch.zeros(total["f64"], dtype=torch.float64, device="cuda"),
                            f32c=torch.zeros(total["f32c"], dtype=torch.float32, device="cuda"),
                            rows=torch.zeros(row, phtl.MON_FIELDS, dtype=torch.float64, device="cuda"))
        jobs = []
        for j, c in zip(plan, start):
            flat, bufs = state["out"][j["dtype"]], []
            for i in range(2):
                a = _pack(c[i], j["dtype"])
                at = j["at"] + i * _slot(j)
                bufs.append(flat[at:at + a.numel()].copy_(a))
            jobs.append(phtl.make_job(*bufs, turns=j["turns"], voltage_V=j["voltage"],
                                      integrator=j["scheme"], dtype=j["dtype"],
                                      monitor=state["out"]["rows"][j["row"]:j["row"] + j["turns"] + 1]))
        state["batch"] = phtl.Batch(R, jobs)
        return state
    state["bufs"] = [[_pack(a, case["dtype"]) for a in c] for c in start]
    state["mon"] = [_rows(case["turns"], case["stride"]) if case["stride"] else None for _ in start]
    if kind == "host":
        state["bufs"] = [[None if a is None else a.cpu().pin_memory() for a in c] for c in state["bufs"]]
        state["mon"] = [None if m is None else m.cpu().pin_memory() for m in state["mon"]]
    if kind == "ramp":
        R.set_programme(*_programme(case))
    if kind == "collective":
        R.set_wake(_wake(case), WAKE_LO, WAKE_HI, WAKE_ALPHA, WAKE_SC)
    if kind != "host" and kind != "schemes" and case["stride"]:
        R.set_monitor(state["mon"][0], stride=case["stride"])
    return state


def run(state):
    case, R = state["case"], state["ring"]
    kind = case["kind"]
    if kind == "batch":
        state["batch"].run()
        return state["out"]
    if kind == "schemes":
        for s, b, m in zip(SCHEMES, state["bufs"], state["mon"]):
            R.set_monitor(m, stride=case["stride"])
            R.track(*b, turns=case["turns"], integrator=s, dtype=case["dtype"])
    else:
        b, m = state["bufs"][0], state["mon"][0]
        opt = dict(turns=case["turns"], integrator=case["scheme"], dtype=case["dtype"])
        if kind == "host":
            R.track_host(*b, mon_rows=m, mon_stride=max(1, case["stride"]), **opt)
        elif kind == "ramp":
            R.track_programme(*b, turn0=0, **opt)
        elif kind == "collective":
            R.track_collective(*b, **opt)
        else:
            R.track(*b, **opt)
    return [a for b, m in zip(state["bufs"], state["mon"]) for a in b + [m] if a is not None]


# ---- work ------------------------------------------------------------------------------

def _flops_per_turn(case, scheme=None, planes=None):
    """Operations of the method per particle and turn (a fused multiply-add is 2): a drift 2
    (6 with the slippage expansion), a kick 25 with its sine at 20 (another 25 with a second RF
    system), a plane 6 (41 where it is chromatic), the ramp's three products."""
    scheme = scheme or case["scheme"]
    planes = case["planes"] if planes is None else planes
    wide, dual = case.get("map") == "widened", case.get("map") == "dual"
    kicks = {"euler_cromer": 1, "leapfrog": 1, "ruth4": 3, "rk4": 4}[scheme]
    drifts = {"euler_cromer": 1, "leapfrog": 2, "ruth4": 4, "rk4": 4}[scheme]
    f = kicks * (50 if dual else 25) + drifts * (6 if wide else 2) + planes * (41 if wide else 6)
    if scheme == "rk4":
        f += 26
    return f + (3 if case["kind"] in ("ramp", "collective") else 0)


def work(case):
    if case["kind"] == "batch":
        jobs = _batch_jobs(case)
        plain = dict(kind="track", map="linear")
        return dict(bytes=sum(2 * 16 * j["n"] + 128 * (j["turns"] + 1) for j in jobs),
                    flops=sum(j["n"] * j["turns"] * _flops_per_turn(plain, j["scheme"], 0) for j in jobs))
    coords = 2 + 2 * case["planes"]
    runs = SCHEMES if case["kind"] == "schemes" else (case["scheme"],)
    rows = case["turns"] // case["stride"] + 1 if case["stride"] else 0
    return dict(bytes=len(runs) * (2 * 8 * coords * case["n"] + 128 * rows),
                flops=sum(case["n"] * case["turns"] * _flops_per_turn(case, s) for s in runs))


# ---- exact results in 64 bits -----------------------------------------------------------

THETA = 1.0 / (2.0 - 2.0 ** (1.0 / 3.0))
STAGES = {"euler_cromer": (("k", 1.0), ("d", 1.0)),
          "leapfrog": (("d", 0.5), ("k", 1.0), ("d", 0.5)),
          "ruth4": (("d", THETA / 2), ("k", THETA), ("d", (1 - THETA) / 2), ("k", 1 - 2 * THETA),
                    ("d", (1 - THETA) / 2), ("k", THETA), ("d", THETA / 2))}


def _moment_row(c):
    n = c[0].numel()
    row = [torch.full((), float(n), device="cuda", dtype=torch.float64)]
    for a, b in ((c[0], c[1]), (c[2], c[3]), (c[4], c[5])):
        if a is None:
            row += [torch.zeros((), device="cuda", dtype=torch.float64)] * 5
        else:
            row += [a.sum(), b.sum(), (a * a).sum(), (b * b).sum(), (a * b).sum()]
    return torch.stack(row)


def _exact_bunch(c, ring, scheme, turns, stride, voltage=None, case=None):
    """The maps of the library in plain torch on float64 coordinates c (changed in place as a
    list); the rows of raw sums, or None."""
    k, A, eC, _ = _consts(ring, voltage=voltage)
    C = ring["circumference_m"]
    e1, e2 = ring.get("eta1", 0.0) * C, ring.get("eta2", 0.0) * C
    k2 = 2.0 * math.pi * ring.get("harmonic2", 0) / C
    A2 = _consts(ring, voltage=ring["voltage2_V"])[1] if ring.get("voltage2_V") else 0.0
    programme = _programme(case) if case and case["kind"] == "ramp" else None
    slices = case["slices"] if case and case["kind"] == "collective" else 0
    if slices:
        w = torch.tensor(_wake(case), device="cuda", dtype=torch.float64)
        m = torch.arange(slices, device="cuda")
        lag = m[None, :] - m[:, None]
        table = torch.where(lag >= 0, w[lag.clamp(min=0)], torch.zeros((), device="cuda", dtype=torch.float64))
        inv_dz = slices / (WAKE_HI - WAKE_LO)
    rows = [_moment_row(c)] if stride else None
    angle = [2.0 * math.pi * (ring["Qx"] % 1.0), 2.0 * math.pi * (ring["Qy"] % 1.0)]
    xi = [ring.get("xi_x", 0.0), ring.get("xi_y", 0.0)]
    beta = [ring["beta_x_m"], ring["beta_y_m"]]
    phis, sphis, r = 0.0, 0.0, 1.0

    def force(z):
        f = A * (torch.sin(k * z + phis) - sphis)
        return f + A2 * torch.sin(k2 * z) if A2 else f

    def slip(d):
        return ((e2 * d + e1) * d + eC) * d if (e1 or e2) else eC * d

    for t in range(turns):
        z, d = c[0], c[1]
        if programme is not None:
            V, p0 = programme
            _, A, eC, bg = _consts(ring, p0=p0[t], voltage=V[t])
            sphis = (bg / math.sqrt(1.0 + bg * bg)) * (p0[t + 1] - p0[t]) / (ring["charge_e"] * V[t])
            phis, r = math.asin(sphis), p0[t] / p0[t + 1]
        if scheme == "rk4":
            a1, b1 = -slip(d), force(z)
            a2, b2 = -slip(d + 0.5 * b1), force(z + 0.5 * a1)
            a3, b3 = -slip(d + 0.5 * b2), force(z + 0.5 * a2)
            a4, b4 = -slip(d + b3), force(z + a3)
            z, d = z + (a1 + 2 * a2 + 2 * a3 + a4) / 6, d + (b1 + 2 * b2 + 2 * b3 + b4) / 6
        else:
            for what, weight in STAGES[scheme]:
                if what == "k":
                    d = d + weight * force(z)
                else:
                    z = z - weight * slip(d)
        c[0], c[1] = z, d
        for p in range(2):
            u, v = c[2 + 2 * p], c[3 + 2 * p]
            if u is None:
                continue
            if xi[p]:
                mu = angle[p] + (2.0 * math.pi * xi[p]) * d
                cs, sn = torch.cos(mu), torch.sin(mu)
            else:
                cs, sn = math.cos(angle[p]), math.sin(angle[p])
            c[2 + 2 * p], c[3 + 2 * p] = cs * u + beta[p] * sn * v, cs * v - sn / beta[p] * u
        if programme is not None:
            for i in (1, 3, 5):
                if c[i] is not None:
                    c[i] = r * c[i]
        if slices:
            s = torch.floor((c[0] - WAKE_LO) * inv_dz)
            inside = (s >= 0) & (s < slices)
            s = s.clamp(0, slices - 1).long()
            count = torch.bincount(s[inside], minlength=slices).double()
            slope = torch.zeros_like(count)
            slope[1:-1] = 0.5 * (count[2:] - count[:-2])
            slope[0], slope[-1] = count[1] - count[0], count[-1] - count[-2]
            kick = WAKE_ALPHA * (table @ count) + WAKE_SC * slope
            c[1] = torch.where(inside, c[1] + kick[s], c[1])
        if stride and (t + 1) % stride == 0:
            rows.append(_moment_row(c))
    return None if rows is None else torch.stack(rows)


def _lay_out(a, dtype):
    """64-bit values in the layout of run()'s output: heads rounded to float, then the rests."""
    if dtype == "f64":
        return a
    hi = a.float().double()
    return torch.cat([hi, a - hi])


def exact(case, seed):
    start = _inputs(case, seed)
    if case["kind"] == "batch":
        parts, rows = dict(f64=[], f32c=[]), []
        for j, c in zip(_batch_jobs(case), start):
            c = [_unpack(_pack(a, j["dtype"]), j["dtype"]) for a in c]
            rows.append(_exact_bunch(c, dict(RING, voltage_V=VOLTAGE), j["scheme"], j["turns"], 1,
                                     voltage=j["voltage"]))
            for a in c[:2]:
                slot = torch.zeros(_slot(j), dtype=torch.float64, device="cuda")
                a = _lay_out(a, j["dtype"])
                slot[:a.numel()] = a
                parts[j["dtype"]].append(slot)
        none = torch.zeros(0, dtype=torch.float64, device="cuda")
        return dict(f64=torch.cat(parts["f64"] + [none]), f32c=torch.cat(parts["f32c"] + [none]),
                    rows=torch.cat(rows))
    out = []
    for i, c in enumerate(start):
        c = [_unpack(_pack(a, case["dtype"]), case["dtype"]) for a in c]
        rows = _exact_bunch(c, _ring(case), SCHEMES[i] if case["kind"] == "schemes" else case["scheme"],
                            case["turns"], case["stride"], case=case)
        out += [_lay_out(a, case["dtype"]) for a in c if a is not None] + ([] if rows is None else [rows])
    return out
