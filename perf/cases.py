"""The calls whose time matters to a user of this library, as cases that a timing program can run.

A case is a dict of plain values; ``prepare`` makes its inputs on the GPU from a seed, ``run`` makes
one pass through the package's public entry points, ``exact`` restates the computation in 64-bit
torch without the package, and ``work`` counts what the computation cannot do without.

Inputs are simulated tracks in the detector of the repository's benchmark: a barrel of ten layers of
flat silicon modules and seven endcap disks a side (34,628 surfaces), or a telescope of nine planes;
a 2 T field along z, or the r-z map of a finite solenoid. Each simulated particle scatters and loses
energy in every module it crosses, and its hits are smeared by 10 um.
"""

import math
import random

import numpy as np
import torch

import paper_2505_22822_gb300 as tkf
from paper_2505_22822_gb300 import learn

KAPPA = 2.99792458e-4  # GeV / (T mm)
ELECTRON, MUON, PION = 0.51099895e-3, 0.1056583755, 0.13957039  # GeV
THICKNESS, X0 = 0.3, 93.7  # mm of silicon
MAX_HITS = 18
HOLE = 1 << 31
TOL, H_MAX, SURF_TOL = 1e-4, 1000.0, 1e-2  # the library's step control defaults


# ---------------------------------------------------------------------------- cases
def listed():
    return [
        # The smallest call: the telescope of the repository's smoke run, FP64, library defaults.
        _fit("telescope_fp64_1k", 1000, detector="telescope"),
        # One event of a trigger process: host buffers in, fitted tracks out, mixed precision.
        _fit("event_host_mixed_5k", 5000, precision="mixed", host=True),
        # The benchmark's batch (50 events in one launch) in plain FP64, launch shape tuned.
        _fit("batch_fp64_600k", 600_000, tuned=True),
        # The same batch as the throughput headline: mixed precision with the learned first step.
        _fit("batch_learned_600k", 600_000, precision="mixed", learned=True, tuned=True),
        # Muons through the solenoid's field map in mixed precision, and the FP64 fit of the same.
        _fit("map_mixed_100k", 100_000, precision="mixed", field="map", tuned=True),
        _fit("map_fp64_50k", 50_000, field="map"),
        # The optimal (two-filter) smoother instead of RTS.
        _fit("two_filter_mixed_200k", 200_000, precision="mixed", smoother="two_filter", tuned=True),
        # Every entry's smoothed state (alignment, residual studies), a tenth of the entries holes.
        _fit("states_mixed_100k", 100_000, precision="mixed", states=True, holes=0.1),
        # Track finding: five dense events in one launch in mixed precision, and one ordinary event in
        # the default FP64.
        _find("find_mixed_80k", 80_000, events=5, precision="mixed"),
        _find("find_fp64_10k", 10_000, events=1),
        # Seed parameters from three measurements of every track of the benchmark's batch.
        {"name": "seeds_600k", "kind": "seeds", "n": 600_000, "field": "uniform", "which": "first_middle_last"},
        # Training of the step proposer: two epochs over the benchmark's number of step records.
        {"name": "train_380k", "kind": "train", "n": 380_000, "batch": 1024, "epochs": 2},
    ]


def _fit(name, n, detector="barrel", field="uniform", precision="fp64", smoother="rts", learned=False, states=False,
         holes=0.0, host=False, tuned=False):
    c = {"kind": "fit", "n": n, "detector": detector, "field": field, "precision": precision, "smoother": smoother,
         "learned": learned, "states": states, "holes": holes, "host": host, "tuned": tuned}
    return dict(c, name=name) if name else c


def _find(name, n, events, precision="fp64", field="uniform", beam=3):
    c = {"kind": "find", "n": n, "events": events, "precision": precision, "field": field, "beam": beam}
    return dict(c, name=name) if name else c


def draw(rng: random.Random):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["telescope", "plain", "plain", "learned", "map", "two_filter", "states", "find", "seeds", "train"])
    precision = rng.choice(["fp64", "mixed"])
    field = rng.choice(["uniform", "uniform", "map"])
    if kind == "telescope":
        return _fit(None, size(300, 20_000), detector="telescope", precision=precision)
    if kind == "plain":
        host = rng.random() < 0.3
        return _fit(None, size(500, 200_000 if host else 600_000), precision=precision, host=host, tuned=rng.random() < 0.5,
                    holes=rng.choice([0.0, 0.0, 0.1]))
    if kind == "learned":
        return _fit(None, size(2000, 600_000), precision="mixed", learned=True, tuned=rng.random() < 0.5)
    if kind == "map":
        return _fit(None, size(500, 60_000 if precision == "fp64" else 200_000), precision=precision, field="map")
    if kind == "two_filter":
        return _fit(None, size(1000, 100_000), precision=precision, smoother="two_filter", field=field)
    if kind == "states":
        return _fit(None, size(500, 100_000), precision=precision, states=True, field=field, holes=rng.choice([0.0, 0.1]))
    if kind == "find":
        events = rng.randint(1, 4)
        return _find(None, size(300 * events, 8000 * events), events, precision, beam=rng.choice([1, 3]))
    if kind == "seeds":
        return {"kind": "seeds", "n": size(1000, 600_000), "field": field,
                "which": rng.choice(["first_middle_last", "first_three"])}
    return {"kind": "train", "n": size(20_000, 380_000), "batch": rng.choice([512, 1000, 1024, 4096]), "epochs": 1}


# ---------------------------------------------------------------------------- detector
_kept = {}


def _keep(key, make):
    """What a program makes once and keeps: the library context, geometries, fields, weights."""
    if key not in _kept:
        _kept[key] = make()
    return _kept[key]


def _context():
    return _keep("context", lambda: tkf.Context(0))


def _telescope_table():
    t = np.zeros((9, 14))
    t[:, 1] = t[:, 5] = t[:, 6] = 1.0  # u = y, v = z, n = x
    t[:, 9] = 50.0 * np.arange(9)
    t[:, 12], t[:, 13] = THICKNESS, X0
    return t, np.zeros((0, 8)), np.zeros((0, 4))


def _barrel_table():
    """Surface table [n, 14] (u v n c thickness x0), layer rows and ring rows."""
    rows, layers, rings, first = [], [], [], 0

    def block(u, v, c):
        n = np.cross(u, v)
        rows.append(np.concatenate([u, v, n, c, np.full((len(u), 1), THICKNESS), np.full((len(u), 1), X0)], 1))

    for i in range(10):
        r = 32.0 * (1000.0 / 32.0) ** (i / 9.0)
        nphi = math.ceil(2 * math.pi * r / 28.0)
        iz, ip = np.divmod(np.arange(18 * nphi), nphi)
        phi = 2 * np.pi * ip / nphi
        cp, sp, zero = np.cos(phi), np.sin(phi), np.zeros(len(phi))
        rr = r + (ip + iz) % 2
        block(np.stack([-sp, cp, zero], 1), np.stack([zero, zero, zero + 1], 1),
              np.stack([rr * cp, rr * sp, (iz - 8.5) * 68.0], 1))
        layers.append([0, r, nphi, 18, 68.0, first, 15.0, 35.0])
        first += len(phi)
    for sign in (-1.0, 1.0):
        for j in range(7):
            z = sign * (600.0 + 400.0 * j)
            layers.append([1, z, 15, len(rings), 68.0, 32.0, 35.0, 15.0])
            for k in range(15):
                rc = 32.0 + 68.0 * k + 35.0
                nphi = math.ceil(2 * math.pi * rc / 28.0)
                ip = np.arange(nphi)
                phi = 2 * np.pi * ip / nphi
                cp, sp, zero = np.cos(phi), np.sin(phi), np.zeros(nphi)
                block(np.stack([cp, sp, zero], 1), np.stack([-sp, cp, zero], 1),
                      np.stack([rc * cp, rc * sp, z + sign * ((ip + k) % 2)], 1))
                rings.append([rc, nphi, first, 0])
                first += nphi
    return np.concatenate(rows), np.array(layers, np.float64), np.array(rings, np.float64)


def _tables(detector):
    return _keep(("tables", detector), _telescope_table if detector == "telescope" else _barrel_table)


def _surfaces(detector):
    """The surface table on the GPU, [14, n]."""
    return _keep(("surf", detector), lambda: torch.from_numpy(np.ascontiguousarray(_tables(detector)[0].T)).cuda())


def _geometry(detector):
    def make():
        table, layers, rings = _tables(detector)
        geo = tkf.Geometry.from_table(_context(), table)
        return geo if detector == "telescope" else geo.set_layers(layers, rings)
    return _keep(("geo", detector), make)


def _solenoid():
    """(B_r, B_z) [nz, nr] float32 of an ideal solenoid (radius 1.2 m, length 5.8 m, 2 T at the centre) by
    the closed form of Derby and Olbert with Bulirsch's complete elliptic integral, every 5 mm."""
    def cel(kc, p, c, s):
        p = np.sqrt(p)
        s = s / p
        f, em, kk = c, 1.0, kc
        c, g = c + s / p, kc / p
        s, p = 2 * (s + f * g), g + p
        em = kc + em
        for _ in range(14):
            k = 2 * np.sqrt(kk)
            kk, f = k * em, c
            c, g = c + s / p, kk / p
            s, p = 2 * (s + f * g), g + p
            em = k + em
        return 0.5 * np.pi * (s + c * em) / (em * (em + p))

    a, b = 1200.0, 2900.0

    def field(rho, z):
        br = bz = 0.0
        gamma = (a - rho) / (a + rho)
        for sign in (1.0, -1.0):
            zz = z + sign * b
            d2 = zz * zz + (rho + a) ** 2
            kc = np.sqrt((zz * zz + (a - rho) ** 2) / d2)
            br = br + sign * a / np.sqrt(d2) * cel(kc, 1.0, 1.0, -1.0)
            bz = bz + sign * zz / np.sqrt(d2) * a / (a + rho) * cel(kc, gamma * gamma, 1.0, gamma)
        return br, bz

    r = np.minimum(5.0 * np.arange(241), a * (1 - 1e-6))
    z = -3500.0 + 5.0 * np.arange(1401)
    br, bz = field(r[None, :], z[:, None])
    scale = 2.0 / field(np.zeros(1), np.zeros(1))[1][0]
    br[:, 0] = 0.0
    return (br * scale).astype(np.float32), (bz * scale).astype(np.float32)


def _field(kind):
    def make():
        if kind == "uniform":
            return tkf.Field.uniform(_context(), (0.0, 0.0, 2.0))
        return tkf.Field.rz_grid(_context(), *_keep("solenoid", _solenoid), 0.0, 5.0, -3500.0, 5.0)
    return _keep(("field", kind), make)


def _field_at(kind):
    """x [3, n] -> B [3, n], FP64; the map is the bilinear interpolation of its FP32 nodes."""
    if kind == "uniform":
        return lambda x: torch.stack([torch.zeros_like(x[0]), torch.zeros_like(x[0]), torch.full_like(x[0], 2.0)])
    br, bz = _keep("solenoid_gpu", lambda: [torch.from_numpy(f).cuda().double() for f in _keep("solenoid", _solenoid)])

    def at(x):
        r = torch.hypot(x[0], x[1])
        fr, fz = r / 5.0, (x[2] + 3500.0) / 5.0
        out = (fr > 240) | (fz < 0) | (fz > 1400)
        i, j = (torch.nan_to_num(f, nan=0.0).clamp(0, top).long() for f, top in ((fr, 239.0), (fz, 1399.0)))
        a, b = fr - i, fz - j
        lo = [(1 - a) * f[j, i] + a * f[j, i + 1] for f in (br, bz)]
        hi = [(1 - a) * f[j + 1, i] + a * f[j + 1, i + 1] for f in (br, bz)]
        rr, zz = (torch.where(out, 0.0, (1 - b) * p + b * q) for p, q in zip(lo, hi))
        s = torch.where(r > 0, rr / r, 0.0)
        return torch.stack([s * x[0], s * x[1], zz])
    return at


# ---------------------------------------------------------------------------- simulation
def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]])


def _bethe(p, mass):
    """Mean energy loss in silicon, GeV/mm (PDG, density effect by its high-energy asymptote)."""
    e = torch.sqrt(p * p + mass * mass)
    beta2, bg2 = (p / e) ** 2, (p / mass) ** 2
    wmax = 2 * ELECTRON * bg2 / (1 + 2 * (e / mass) * ELECTRON / mass + (ELECTRON / mass) ** 2)
    half_delta = (math.log(31.05 / 173.0) + 0.5 * torch.log(bg2) - 0.5).clamp(min=0.0)
    bracket = 0.5 * torch.log(2 * ELECTRON * bg2 * wmax / 173e-9 ** 2) - beta2 - half_delta
    return 0.307075 * 0.49848 / beta2 * bracket * 2.329 * 1e-4


def _highland(p, mass, xx0):
    """Projected scattering angle."""
    beta2 = p * p / (p * p + mass * mass)
    return 0.0136 / (torch.sqrt(beta2) * p) * torch.sqrt(xx0) * (1 + 0.038 * torch.log(xx0 / beta2))


def _crossed(n, gen, field):
    """Particles from the beam line and the modules they cross, in order: vertex z, phi, theta, q/p and
    module ids [n, 18] (-1: none), at least six a particle."""
    _, layers, rings = _tables("barrel")
    z0, phi, theta, qop, ids = [], [], [], [], []
    have = 0
    while have < n:
        m = int(1.2 * (n - have)) + 64
        u = torch.rand(4, m, generator=gen, device="cuda", dtype=torch.float64)
        zv = 50.0 * torch.randn(m, generator=gen, device="cuda", dtype=torch.float64)
        th = 2 * torch.atan(torch.exp(3.0 - 6.0 * u[0]))
        ph = 2 * math.pi * u[1]
        q = torch.where(u[2] < 0.5, -1.0, 1.0)
        # pions with pT log-uniform 0.5-100 GeV, or in the map muons with p log-uniform 1-100 GeV
        pt = 0.5 * 200.0 ** u[3] if field == "uniform" else 100.0 ** u[3] * torch.sin(th)
        radius = pt / (KAPPA * 2.0)
        cot = torch.cos(th) / torch.sin(th)
        arc = torch.full((m, len(layers)), math.inf, device="cuda", dtype=torch.float64)
        mid = torch.full((m, len(layers)), -1, device="cuda", dtype=torch.int64)
        # arc length where a particle leaves the detector
        reach = 2 * radius * torch.asin((1050.0 / (2 * radius)).clamp(max=1.0))
        two_pi = 2 * math.pi
        for li, lay in enumerate(layers):
            if lay[0] == 0:
                ok = 2 * radius > lay[1]
                turn = 2 * torch.asin((lay[1] / (2 * radius)).clamp(max=1.0))
                s = radius * turn
                az = (ph - q * 0.5 * turn) % two_pi
                iz = torch.floor((zv + s * cot) / 68.0 + 9.0)
                ok &= (iz >= 0) & (iz < 18)
                idx = lay[5] + iz * lay[2] + torch.round(az * (lay[2] / two_pi)) % lay[2]
            else:
                s = (lay[1] - zv) / cot
                turn = s / radius
                az = (ph - q * 0.5 * turn) % two_pi
                k = torch.floor((2 * radius * torch.sin(0.5 * turn) - 32.0) / 68.0)
                ok = (s > 0) & (s < reach) & (k >= 0) & (k < 15)
                row = int(lay[3]) + torch.nan_to_num(k, nan=0.0).clamp(0, 14).long()
                rg = _keep("rings", lambda: torch.from_numpy(rings).cuda())[row]
                idx = rg[:, 2] + torch.round(az * (rg[:, 1] / two_pi)) % rg[:, 1]
            mid[:, li] = torch.where(ok, idx.long(), -1)
            # the flat module's plane lies a little before or after the layer's nominal surface
            rec = _surfaces("barrel")[:, mid[:, li].clamp(min=0)]
            r = 2 * radius * torch.sin(0.5 * turn)
            x = torch.stack([r * torch.cos(az), r * torch.sin(az), zv + s * cot])
            T = torch.stack([torch.cos(ph - q * turn), torch.sin(ph - q * turn), cot])
            arc[:, li] = torch.where(ok, s + _dot(rec[6:9], rec[9:12] - x) / _dot(rec[6:9], T), math.inf)
        order = torch.argsort(arc, dim=1, stable=True)[:, :MAX_HITS]
        mid = torch.gather(mid, 1, order)
        keep = ((mid >= 0).sum(1) >= 6).nonzero()[: n - have, 0]
        for to, x in zip((z0, phi, theta, qop, ids), (zv, ph, th, q * torch.sin(th) / pt, mid)):
            to.append(x[keep])
        have += len(keep)
    return [torch.cat(x) for x in (z0, phi, theta, qop, ids)]


def _fly(field, x, T, qop, surf):
    """Position and direction where the particle meets the plane: fourth-order Runge-Kutta along the
    path, in pieces of the parabola's length to the plane."""
    c, nrm = surf[9:12], surf[6:9]

    def rk(x, T, h):
        def f(x, T):
            return KAPPA * qop * _cross(T, field(x))
        k1 = f(x, T)
        k2 = f(x + 0.5 * h * T + 0.125 * h * h * k1, T + 0.5 * h * k1)
        k3 = f(x + 0.5 * h * T + 0.125 * h * h * k1, T + 0.5 * h * k2)
        k4 = f(x + h * T + 0.5 * h * h * k3, T + h * k3)
        x = x + h * T + h * h / 6 * (k1 + k2 + k3)
        T = T + h / 6 * (k1 + 2 * k2 + 2 * k3 + k4)
        return x, T / torch.sqrt(_dot(T, T))

    for left in (4, 3, 2, 1, 1, 1):
        d, a = _dot(nrm, c - x), _dot(nrm, T)
        b = _dot(nrm, KAPPA * qop * _cross(T, field(x)))
        disc = a * a + 2 * b * d
        s = torch.where(disc > 0, 2 * d / (a + torch.copysign(torch.sqrt(disc.clamp(min=0)), a)), d / a)
        x, T = rk(x, T, s / left)
    s = _dot(nrm, c - x) / _dot(nrm, T)
    return x + s * T, T


def _tracks(case, seed):
    """Simulated tracks in the library's batch layout (CUDA tensors), with ids [n, 18] of the crossings."""
    n, detector, kind = case["n"], case.get("detector", "barrel"), case["field"]
    gen = torch.Generator(device="cuda").manual_seed(seed)
    surf, field = _surfaces(detector), _field_at(kind)

    def normal(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=torch.float64)

    if detector == "telescope":  # muons of 1-10 GeV within 0.1 rad of the axis
        u = torch.rand(4, n, generator=gen, device="cuda", dtype=torch.float64)
        az, dip = 0.2 * u[0] - 0.1, 0.2 * u[1] - 0.1
        T = torch.stack([torch.cos(dip) * torch.cos(az), torch.cos(dip) * torch.sin(az), torch.sin(dip)])
        x = torch.zeros_like(T)
        qop = torch.where(u[3] < 0.5, -1.0, 1.0) / (1.0 + 9.0 * u[2])
        ids = torch.arange(9, device="cuda").expand(n, 9)
        mass = MUON
    else:
        z0, phi, theta, qop, ids = _crossed(n, gen, kind)
        if case.get("states"):  # some last hits lost: the outputs' size depends on n alone
            lost = int((ids >= 0).sum()) - int(9.8 * n)
            while lost > 0:
                count = (ids >= 0).sum(1)
                cut = count > 6
                cut &= torch.cumsum(cut, 0) <= lost
                ids[cut, count[cut] - 1] = -1
                lost -= int(cut.sum())
        T = torch.stack([torch.sin(theta) * torch.cos(phi), torch.sin(theta) * torch.sin(phi), torch.cos(theta)])
        x = torch.stack([torch.zeros_like(z0), torch.zeros_like(z0), z0])
        mass = MUON if kind == "map" else PION
    loc, seed_par = torch.zeros(2, *ids.shape, device="cuda", dtype=torch.float64), None
    for k in range(ids.shape[1]):
        live = ids[:, k] >= 0
        s = surf[:, ids[:, k].clamp(min=0)]
        xn, Tn = _fly(field, x, T, qop, s)
        x, T = torch.where(live, xn, x), torch.where(live, Tn, T)
        for j in (0, 1):
            loc[j, :, k] = _dot(s[3 * j:3 * j + 3], x - s[9:12])
        if k == 0:
            seed_par = torch.stack([loc[0, :, 0], loc[1, :, 0], torch.atan2(T[1], T[0]), torch.acos(T[2]), qop])
        # scattering and energy loss in the module
        path = THICKNESS / _dot(s[6:9], T).abs()
        p = 1 / qop.abs()
        th0 = _highland(p, mass, path / X0)
        st = torch.sqrt(T[0] ** 2 + T[1] ** 2)
        e1 = torch.stack([T[2] * T[0] / st, T[2] * T[1] / st, -st])
        e2 = torch.stack([-T[1] / st, T[0] / st, torch.zeros_like(st)])
        g = normal(2, n)
        Ts = T + th0 * (g[0] * e1 + g[1] * e2)
        T = torch.where(live, Ts / torch.sqrt(_dot(Ts, Ts)), T)
        e = torch.sqrt(p * p + mass * mass) - _bethe(p, mass) * path
        qop = torch.where(live, torch.copysign(1 / torch.sqrt((e * e - mass * mass).clamp(min=1e-4)), qop), qop)
    loc = loc + 0.01 * normal(2, *ids.shape)
    # seed: the truth at the first module smeared like a seed of three hits
    sth = torch.sin(seed_par[3])
    sig = torch.stack([sth * 0 + 0.05, sth * 0 + 0.05, sth * 0 + 1e-3, 1e-3 * sth * sth, 0.1 * seed_par[4].abs()])
    if detector == "telescope":
        sig = torch.stack([sth * 0 + 1.0, sth * 0 + 1.0, sth * 0 + 0.01, sth * 0 + 0.01, 0.1 * seed_par[4].abs()])
    seed_par = seed_par + sig * normal(5, n)
    seed_par[2] = torch.remainder(seed_par[2] + math.pi, 2 * math.pi) - math.pi
    seed_cov = torch.zeros(15, n, device="cuda", dtype=torch.float64)
    seed_cov[[0, 5, 9, 12, 14]] = sig * sig
    used = ids >= 0
    sid = ids[used]
    if case.get("holes", 0.0) > 0.0:  # a crossed module without a hit
        hole = torch.rand(ids.shape, generator=gen, device="cuda") < case["holes"]
        hole[:, 0] = False
        sid = torch.where(hole[used], sid + HOLE, sid)
    offsets = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
    offsets[1:] = torch.cumsum(used.sum(1), 0)
    var = torch.full((len(sid),), 1e-4, device="cuda", dtype=torch.float64)
    batch = tkf.Batch(offsets.to(torch.int32), loc[0][used], loc[1][used], var, torch.zeros_like(var), var.clone(),
                      torch.where(sid >= HOLE, sid - (1 << 32), sid).to(torch.int32), seed_par.contiguous(), seed_cov)
    return batch, ids


# ---------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    ctx = _context()
    if case["kind"] == "train":
        return {"case": case, "ctx": ctx, "records": _records(case["n"], seed)}
    detector = case.get("detector", "barrel")
    batch, ids = _tracks(case, seed)
    state = {"case": case, "ctx": ctx, "geo": _geometry(detector), "fld": _field(case["field"]), "batch": batch}
    if case["kind"] == "fit":
        opts = tkf.Options(precision=tkf.MIXED if case["precision"] == "mixed" else tkf.FP64, autotune=case["tuned"],
                           smoother=tkf.SMOOTHER_TWO_FILTER if case["smoother"] == "two_filter" else tkf.SMOOTHER_RTS)
        if case["learned"]:
            opts.step_mode = tkf.STEP_LEARNED
            opts.mlp = _keep("mlp", lambda: tkf.Mlp(ctx, _proposer()))
        state["opts"] = opts
        if case["host"]:
            state["batch"] = batch.to("cpu").to("cpu", pin=True)
            out = tkf.alloc_outputs(case["n"], "cpu")
            state["out"] = tkf.Result(*(x.pin_memory() if x is not None else None for x in vars(out).values()))
    elif case["kind"] == "find":
        state["event"] = _event(case, batch, ids, seed)
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "train":
        params, loss = learn.train(ctx, state["records"], epochs=case["epochs"], batch=case["batch"])
        return {"params": params, "loss": loss}
    geo, fld, batch = state["geo"], state["fld"], state["batch"]
    if case["kind"] == "seeds":
        which = tkf.SEED_FIRST_THREE if case["which"] == "first_three" else tkf.SEED_FIRST_MIDDLE_LAST
        s = tkf.estimate_seeds(ctx, geo, fld, batch, which)
        return {"par": s.par, "cov": s.cov, "status": s.status}
    if case["kind"] == "find":
        opts = tkf.Options(precision=tkf.MIXED if case["precision"] == "mixed" else tkf.FP64)
        r = tkf.find_tracks(ctx, geo, fld, *state["event"][:-1], opts, beam=case["beam"], seed_event=state["event"][-1])
        return {"n_entries": r.n_entries, "n_meas": r.n_meas, "chi2": r.chi2, "sid": r.entry_sid, "meas": r.entry_meas}
    if case["host"]:
        r = tkf.fit_host(ctx, geo, fld, batch, state["opts"], out=state["out"])
    else:
        r = tkf.fit(ctx, geo, fld, batch, state["opts"], states=case["states"])
    out = {"par": r.par, "cov": r.cov, "chi2": r.chi2, "ndf": r.ndf, "status": r.status, "steps": r.steps}
    if case["states"]:
        out.update(states_par=r.states_par, states_cov=r.states_cov)
    return out


def _event(case, batch, ids, seed):
    """find_tracks' arguments: seeds (every particle's first module and smeared parameters) and the events'
    measurements by surface, a tenth of them noise."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1)
    n, n_surf = case["n"], _surfaces("barrel").shape[1]
    event = (torch.arange(n, device="cuda") * case["events"]) // n
    m = len(batch.loc0)
    per_hit = torch.repeat_interleave(event, (ids >= 0).sum(1))
    pick = torch.randint(0, m, (m // 10,), generator=gen, device="cuda")
    noise = torch.rand(2, len(pick), generator=gen, device="cuda", dtype=torch.float64) * 30.0 - 15.0
    sid = torch.cat([batch.sid, batch.sid[pick]]).long()
    key = torch.cat([per_hit, per_hit[pick]]) * n_surf + sid
    order = torch.argsort(key, stable=True)
    counts = torch.bincount(key, minlength=case["events"] * n_surf)
    ends = torch.cumsum(counts, 0).reshape(case["events"], n_surf)
    offsets = torch.cat([torch.cat([ends.new_zeros(1), ends[:-1, -1]])[:, None], ends], 1).to(torch.int32).contiguous()
    loc = [torch.cat([x, y])[order].contiguous() for x, y in zip((batch.loc0, batch.loc1), noise)]
    var = torch.full((len(order),), 1e-4, device="cuda", dtype=torch.float64)
    first = batch.sid[batch.offsets[:-1].long()].contiguous()
    return [first, batch.seed_par, batch.seed_cov, offsets, *loc, var, torch.zeros_like(var), var.clone(),
            event.to(torch.int32)]


def _records(n, seed):
    """Step records [n, 13]: the twelve network inputs and ln of the largest step within tolerance."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand(8, n, generator=gen, device="cuda", dtype=torch.float64)
    theta = 2 * torch.atan(torch.exp(3.0 - 6.0 * u[0]))
    qop = torch.sin(theta) / (0.5 * 200.0 ** u[1]) * torch.where(u[2] < 0.5, -1.0, 1.0)
    az = 0.6 * u[3] - 0.3
    gap = 0.01 + 0.3 * u[4]
    b = KAPPA * 2.0 * qop.abs()
    label = 0.25 * torch.log(4 * TOL / (b ** 3 * torch.sin(theta) * (az.cos() + az.sin().abs())))
    zero = torch.zeros_like(u[0])
    return torch.stack([0.03 * u[5] - 0.015, 0.07 * u[6] - 0.035, -gap, torch.sin(theta) * torch.sin(az), torch.cos(theta),
                        torch.sin(theta) * torch.cos(az), qop, zero, zero, zero + 1.0, label * 0.2 + 0.1 * u[7],
                        (gap / (torch.sin(theta) * torch.cos(az))).clamp(max=2.0), label], 1).float().contiguous()


def _proposer():
    """BF16 weights of a step proposer, as a program would load them: two random layers and an output layer
    fitted to the largest step within tolerance, shifted so that few proposals exceed it."""
    rng = np.random.default_rng(7)
    rec = _records(20_000, 7).double().cpu().numpy()

    def bf16(x):
        u = np.ascontiguousarray(x, np.float32).view(np.uint32)
        return ((u + 0x7FFF + ((u >> 16) & 1)) >> 16).astype(np.uint16)

    def silu(z):
        return z / (1 + np.exp(-z))

    rec[:, 10] = 0.2 * np.log(H_MAX)
    w1 = rng.normal(size=(64, 12)) * np.array([1, 1, 1, 1, 1, 1, 3, 0, 0, 0.1, 0.1, 0.5])
    b1, w2, b2 = rng.normal(size=64), rng.normal(size=(64, 64)) / 6, 0.5 * rng.normal(size=64)
    a = silu(silu(rec[:, :12] @ w1.T + b1) @ w2.T + b2)
    a1 = np.concatenate([a, np.ones((len(a), 1))], 1)
    w3 = np.linalg.solve(a1.T @ a1 + 1e-2 * np.eye(65), a1.T @ rec[:, 12])
    w3[64] += np.quantile(rec[:, 12] - a1 @ w3, 0.05)
    return bf16(np.concatenate([w1.ravel(), b1, w2.ravel(), b2, w3]))


# ---------------------------------------------------------------------------- 64-bit restatement
def exact(case, seed):
    if case["kind"] == "train":
        return _exact_train(case, seed)
    if case["kind"] == "find":
        return None  # a search whose result is whole numbers; a plain torch search of the events takes minutes
    batch, _ = _tracks(case, seed)
    if case["kind"] == "seeds":
        return _exact_seeds(case, batch)
    return _exact_fit(case, batch)


def _exact_train(case, seed):
    """The same regression without the operands' BF16 rounding."""
    rec = _records(case["n"], seed)
    gen = torch.Generator(device="cuda").manual_seed(7)
    rec = rec[torch.randperm(case["n"], device="cuda", generator=gen)].double()
    # seeded initial weights: SplitMix64 of (seed, index), uniform within 1/sqrt(fan in), biases 0
    with np.errstate(over="ignore"):
        k = np.arange(5057, dtype=np.uint64)
        x = np.uint64(7) * np.uint64(0x100000001B3) + k + np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        x = x ^ (x >> np.uint64(31))
    fan = np.where(k < 768, 12.0, 64.0)
    weight = (k < 768) | ((k >= 832) & (k < 4928)) | ((k >= 4992) & (k < 5056))
    p = torch.from_numpy(np.where(weight, (2 * (x >> np.uint64(40)).astype(np.float64) / 2 ** 24 - 1) / np.sqrt(fan), 0)).cuda()
    m, v = torch.zeros_like(p), torch.zeros_like(p)
    losses, step = [], 0
    for _ in range(case["epochs"]):
        total = 0.0
        for i in range(case["n"] // case["batch"]):
            part = rec[i * case["batch"]:(i + 1) * case["batch"]]
            w = p.clone().requires_grad_(True)
            z = torch.nn.functional.silu(part[:, :12] @ w[:768].view(64, 12).T + w[768:832])
            z = torch.nn.functional.silu(z @ w[832:4928].view(64, 64).T + w[4928:4992])
            loss = ((z @ w[4992:5056] + w[5056] - part[:, 12]) ** 2).mean()
            (g,) = torch.autograd.grad(loss, w)
            step += 1
            m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
            p = p - 2e-3 * (m / (1 - 0.9 ** step)) / (torch.sqrt(v / (1 - 0.999 ** step)) + 1e-8)
            total = total + loss.detach()
        losses.append(total / (case["n"] // case["batch"]))
    return {"params": p, "loss": torch.stack(losses)}


def _exact_seeds(case, batch):
    surf, field = _surfaces("barrel"), _field_at(case["field"])
    b0, count = batch.offsets[:-1].long(), (batch.offsets[1:] - batch.offsets[:-1]).long()
    last, middle = (2 + 0 * count, 1 + 0 * count) if case["which"] == "first_three" else (count - 1, (count - 1) // 2)
    rows = [b0, b0 + middle, b0 + last]
    pts, bzs, sh2 = [], [], 0.0
    for m in rows:
        s = surf[:, batch.sid[m].long()]
        pts.append(s[9:12] + batch.loc0[m] * s[0:3] + batch.loc1[m] * s[3:6])
        bzs.append(field(pts[-1])[2])
        sh2 = sh2 + (batch.v00[m] + batch.v11[m]) / 6.0
    bz = (bzs[0] + bzs[1] + bzs[2]) / 3.0
    a, b = pts[1] - pts[0], pts[2] - pts[0]
    a2, b2 = a[0] ** 2 + a[1] ** 2, b[0] ** 2 + b[1] ** 2
    area = 2 * (a[0] * b[1] - a[1] * b[0])
    cx, cy = (b[1] * a2 - a[1] * b2) / area, (a[0] * b2 - b[0] * a2) / area
    radius, turn = torch.hypot(cx, cy), torch.sign(area)
    wx, wy = b[0] - cx, b[1] - cy
    swept = torch.atan2(turn * (cy * wx - cx * wy), -cx * wx - cy * wy) % (2 * math.pi)
    arc = radius * swept
    length = torch.hypot(arc, b[2])
    qop = -turn * torch.sign(bz) * arc / (KAPPA * bz.abs() * radius * length)
    sth = arc / length
    lt2, l2 = b2, b2 + b[2] ** 2
    th0 = 0.0136 * qop.abs() * math.sqrt(THICKNESS / X0) * (1 + 0.038 * math.log(THICKNESS / X0))
    ms2 = last * th0 ** 2
    spread = (torch.stack(bzs).amax(0) - torch.stack(bzs).amin(0)) / bz
    rel2 = (4 * sh2 + ms2 * lt2 / 16) * 64 * radius ** 2 / lt2 ** 2 + spread ** 2 + 1e-4
    cov = torch.zeros(15, len(count), device="cuda", dtype=torch.float64)
    cov[0], cov[1], cov[5] = batch.v00[b0], batch.v01[b0], batch.v11[b0]
    cov[9] = (64 * sh2 / lt2 + 2 * ms2 / sth ** 2 + lt2 / (4 * radius ** 2) * rel2).clamp(max=math.pi ** 2)
    cov[12] = (16 * sh2 / l2 + 2 * ms2).clamp(max=math.pi ** 2)
    cov[14] = rel2 * qop ** 2
    par = torch.stack([batch.loc0[b0], batch.loc1[b0], torch.atan2(-turn * cx, turn * cy), torch.atan2(arc, b[2]), qop])
    return {"par": par, "cov": cov, "status": None}


_UPPER = [(i, j) for i in range(5) for j in range(i, 5)]


def _pack(c):
    return torch.stack([c[:, i, j] for i, j in _UPPER])


def _rkn(field, surf, r, T, lam, dr, dT, h_ctrl):
    """Adaptive Runge-Kutta-Nystrom steps of every track to its plane, with the derivative columns of
    (phi, theta, q/p): dr, dT [3 columns, 3, n]. Tracks that never arrive become NaN."""
    def parabola(d, a, b):
        disc = a * a + 2 * b * d
        q = 2 * d / (a + torch.copysign(torch.sqrt(disc.clamp(min=0)), a))
        return torch.where((disc >= 0) & torch.isfinite(q), q, d / a)

    def columns(T, B, lk, u):
        """Derivative of T x lam kappa B along the columns u of dT (the q/p column has its own source)."""
        q = torch.stack([_cross(u[c], lk * B) for c in range(3)])
        q[2] += _cross(T, KAPPA * B)
        return q

    live = torch.arange(r.shape[1], device=r.device)
    for it in range(400):
        if not len(live):
            break
        s, x, t, l, e, g, hc = surf[:, live], r[:, live], T[:, live], lam[live], dr[:, :, live], dT[:, :, live], h_ctrl[live]
        lk = KAPPA * l
        dist, a = _dot(s[6:9], s[9:12] - x), _dot(s[6:9], t)
        B1 = field(x)
        k1 = _cross(t, lk * B1)
        sp = parabola(dist, a, _dot(s[6:9], k1))
        land = dist.abs() <= SURF_TOL
        if it == 0:
            hc = torch.where(land | (dist / a > -1.0), hc, math.nan)
        limited = ~(sp.abs() < hc)
        h = torch.where(limited, torch.copysign(hc, sp), sp)
        B2 = field(x + 0.5 * h * t + 0.125 * h * h * k1)
        T2 = t + 0.5 * h * k1
        k2 = _cross(T2, lk * B2)
        T3 = t + 0.5 * h * k2
        k3 = _cross(T3, lk * B2)
        B4 = field(x + h * t + 0.5 * h * h * k3)
        T4 = t + h * k3
        k4 = _cross(T4, lk * B4)
        eps = h * h * (k1 - k2 - k3 + k4).abs().sum(0)
        fac = torch.where(eps > 0, 0.9 * (TOL / eps) ** 0.25, 4.0).clamp(0.25, 4.0)
        reject = ~land & (eps > TOL)
        step = ~land & ~reject
        q1 = columns(t, B1, lk, g)
        q2 = columns(T2, B2, lk, g + 0.5 * h * q1)
        q3 = columns(T3, B2, lk, g + 0.5 * h * q2)
        q4 = columns(T4, B4, lk, g + h * q3)
        hs = torch.where(step, h, 0.0)
        hl = torch.where(land, sp, 0.0)
        dr[:, :, live] = e + (hs + hl) * g + hs * hs / 6 * (q1 + q2 + q3) + 0.5 * hl * hl * q1
        dT[:, :, live] = g + hs / 6 * (q1 + 2 * q2 + 2 * q3 + q4) + hl * q1
        r[:, live] = x + (hs + hl) * t + hs * hs / 6 * (k1 + k2 + k3) + 0.5 * hl * hl * k1
        T[:, live] = t + hs / 6 * (k1 + 2 * k2 + 2 * k3 + k4) + hl * k1
        h_ctrl[live] = torch.where(reject, h.abs() * fac, torch.where(step & limited, (h.abs() * fac).clamp(max=H_MAX), hc))
        live = live[~land & torch.isfinite(hc)]


def _exact_fit(case, batch):
    """Kalman filter of the muon hypothesis with a textbook Rauch-Tung-Striebel backward pass, or with a
    backward filter of the reversed particle averaged with the seed. Steps start from h_max: another
    accepted step sequence is the same fit within the step tolerance."""
    n = case["n"]
    surf, field = _surfaces(case["detector"]), _field_at(case["field"])
    batch = batch if batch.offsets.is_cuda else batch.to("cuda")
    b0, count = batch.offsets[:-1].long(), (batch.offsets[1:] - batch.offsets[:-1]).long()
    longest = int(count.max())
    eye = torch.eye(5, device="cuda", dtype=torch.float64)

    def unpack(c):
        m = torch.empty(c.shape[1], 5, 5, device="cuda", dtype=torch.float64)
        for x, (i, j) in zip(c, _UPPER):
            m[:, i, j] = m[:, j, i] = x
        return m

    def material(s, T, lam, sign):
        """Highland variance, and q/p after the mean loss (sign -1) or with it given back (+1)."""
        path, p = THICKNESS / _dot(s[6:9], T).abs(), 1 / lam.abs()
        e = torch.sqrt(p * p + MUON * MUON) + sign * _bethe(p, MUON) * path
        return _highland(p, MUON, path / X0) ** 2, torch.copysign(1 / torch.sqrt(e * e - MUON * MUON), lam)

    def scattered(C, th2, theta):
        C = C.clone()
        C[:, 2, 2] += th2 / torch.sin(theta) ** 2
        C[:, 3, 3] += th2
        return C

    def direction(p):
        return torch.stack([torch.sin(p[3]) * torch.cos(p[2]), torch.sin(p[3]) * torch.sin(p[2]), torch.cos(p[3])])

    def transport(p, lam, s0, s1, h_ctrl):
        """Bound parameters on s1 and the Jacobian from those on s0."""
        T = direction(p)
        r = s0[9:12] + p[0] * s0[0:3] + p[1] * s0[3:6]
        sph, cph, sth, cth = torch.sin(p[2]), torch.cos(p[2]), torch.sin(p[3]), torch.cos(p[3])
        zero = torch.zeros_like(sph)
        dT = torch.stack([torch.stack([-sth * sph, sth * cph, zero]), torch.stack([cth * cph, cth * sph, -sth]),
                          torch.stack([zero, zero, zero])])
        dr = torch.zeros_like(dT)
        _rkn(field, s1, r, T, lam, dr, dT, h_ctrl)
        kend = _cross(T, KAPPA * lam * field(r))
        t = T / torch.sqrt(_dot(T, T))
        st = torch.sqrt(t[0] ** 2 + t[1] ** 2)
        J = torch.zeros(len(lam), 5, 5, device="cuda", dtype=torch.float64)
        for c in range(5):
            x = s0[3 * c:3 * c + 3] if c < 2 else dr[c - 2]
            d = torch.zeros_like(T) if c < 2 else dT[c - 2]
            ds = -_dot(s1[6:9], x) / _dot(s1[6:9], T)
            x, d = x + T * ds, d + kend * ds
            J[:, 0, c], J[:, 1, c] = _dot(s1[0:3], x), _dot(s1[3:6], x)
            J[:, 2, c] = (-t[1] * d[0] + t[0] * d[1]) / st ** 2
            J[:, 3, c] = t[2] * (t[0] * d[0] + t[1] * d[1]) / st - st * d[2]
        J[:, 4, 4] = 1.0
        x = r - s1[9:12]
        q = torch.stack([_dot(s1[0:3], x), _dot(s1[3:6], x), torch.atan2(t[1], t[0]), torch.atan2(st, t[2]), lam])
        return q, J

    def update(p, C, m):
        V = torch.stack([torch.stack([batch.v00[m], batch.v01[m]], 1), torch.stack([batch.v01[m], batch.v11[m]], 1)], 1)
        res = torch.stack([batch.loc0[m] - p[0], batch.loc1[m] - p[1]], 1)[:, :, None]
        S = C[:, :2, :2] + V
        Si = torch.stack([torch.stack([S[:, 1, 1], -S[:, 0, 1]], 1), torch.stack([-S[:, 0, 1], S[:, 0, 0]], 1)], 1)
        Si = Si / (S[:, 0, 0] * S[:, 1, 1] - S[:, 0, 1] ** 2)[:, None, None]
        K = C[:, :, :2] @ Si
        A = eye - torch.cat([K, torch.zeros_like(K), torch.zeros_like(K[:, :, :1])], 2)
        hole = (batch.sid[m] < 0)[:, None, None]
        Cn = torch.where(hole, C, A @ C @ A.mT + K @ V @ K.mT)
        pn = torch.where(hole[:, :, 0].T, p, p + (K @ res)[:, :, 0].T)
        return pn, Cn, torch.where(hole[:, 0, 0], 0.0, (res.mT @ Si @ res)[:, 0, 0])

    def wrap(x):
        return torch.remainder(x + math.pi, 2 * math.pi) - math.pi

    def at(k, t):
        return surf[:, (batch.sid[b0[t] + k].long() & 0x7FFFFFFF)]

    p0, C0 = batch.seed_par.clone(), unpack(batch.seed_cov)
    p, C, chi2 = update(p0, C0, b0)
    p[2] = wrap(p[2])
    h_ctrl = torch.full((n,), H_MAX, device="cuda", dtype=torch.float64)
    kept = [(torch.arange(n, device="cuda"), p.clone(), C.clone(), None, None, None)]
    for k in range(1, longest):
        t = (count > k).nonzero()[:, 0]  # tracks with an entry k
        s0, s1, q, h = at(k - 1, t), at(k, t), p[:, t], h_ctrl[t]
        th2, lam = material(s0, direction(q), q[4], -1.0)
        pp, J = transport(q, lam, s0, s1, h)
        Cp = J @ scattered(C[t], th2, q[3]) @ J.mT
        Cp = 0.5 * (Cp + Cp.mT)
        pn, Cn, c2 = update(pp, Cp, b0[t] + k)
        p[:, t], C[t], h_ctrl[t] = pn, Cn, h
        chi2[t] += c2
        kept.append((t, pn, Cn, pp, Cp, J))
    if case["smoother"] == "two_filter":
        flip = torch.tensor([1.0, 1, 1, -1, -1], device="cuda", dtype=torch.float64)
        flips = flip[:, None] * flip[None, :]

        def reverse(p):
            return torch.stack([p[0], p[1], wrap(p[2] + math.pi), math.pi - p[3], -p[4]])

        p, C = reverse(p), 1e3 * flips * C
        for ent in range(longest):
            t = (count > ent).nonzero()[:, 0]
            k = count[t] - 1 - ent
            pp, Cp = p[:, t], C[t]
            if ent:
                h = h_ctrl[t]
                pp, J = transport(pp, pp[4], at(k + 1, t), at(k, t), h)
                h_ctrl[t] = h
                th2, lam = material(at(k, t), direction(pp), pp[4], 1.0)
                pp[4] = lam
                Cp = scattered(J @ Cp @ J.mT, th2, pp[3])
            p[:, t], C[t], _ = update(pp, Cp, b0[t] + k)
        p, C = reverse(p), flips * C
        K = torch.linalg.solve(C + C0, C).mT
        d = p0 - p
        d[2] = wrap(d[2])
        ps = p + (K @ d.T[:, :, None])[:, :, 0].T
        Cs = (eye - K) @ C @ (eye - K).mT + K @ C0 @ K.mT
    else:
        m = len(batch.loc0)
        states = [torch.zeros(j, m, device="cuda", dtype=torch.float64) for j in (5, 15)] if case["states"] else None
        ps, Cs = p.clone(), C.clone()
        for k in range(longest - 1, -1, -1):
            if k + 1 < longest:
                t, _, _, pp, Cp, J = kept[k + 1]
                q, Cf = p_at(kept[k], t), c_at(kept[k], t)
                A = torch.linalg.solve(Cp, J @ Cf).mT
                d = ps[:, t] - pp
                d[2] = wrap(d[2])
                ps[:, t] = q + (A @ d.T[:, :, None])[:, :, 0].T
                Cs[t] = Cf + A @ (Cs[t] - Cp) @ A.mT
            if states:
                t = kept[k][0]
                states[0][:, b0[t] + k], states[1][:, b0[t] + k] = ps[:, t], _pack(Cs[t])
    ps[2] = wrap(ps[2])
    out = {"par": ps, "cov": _pack(Cs), "chi2": chi2, "ndf": None, "status": None, "steps": None}
    if case["states"]:
        states[0][2] = wrap(states[0][2])
        out.update(states_par=states[0], states_cov=states[1])
    return out


def p_at(kept, t):
    """The filtered parameters of tracks t at an entry (its own tracks are sorted and hold all of t)."""
    return kept[1][:, torch.searchsorted(kept[0], t)]


def c_at(kept, t):
    return kept[2][torch.searchsorted(kept[0], t)]


# ---------------------------------------------------------------------------- work
def work(case):
    """Bytes of every input read once and every output written once, and the operations of the method:
    per crossing the transport, update and smoother of a 5 x 5 covariance, per step the four stages."""
    n, hits = case["n"], 9.0 if case.get("detector") == "telescope" else 10.5
    if case["kind"] == "train":
        samples = case["epochs"] * (n // case["batch"]) * case["batch"]
        return {"bytes": samples * 52.0, "flops": samples * 3 * 2.0 * 4928}
    if case["kind"] == "seeds":
        return {"bytes": n * (4 + 3 * 44 + 164.0), "flops": n * 300.0}
    if case["kind"] == "find":
        m = n * hits * 1.1
        return {"bytes": m * 40 + n * (164 + 16 + 24 * 8.0), "flops": n * case["beam"] * hits * 1200.0}
    m = n * hits
    per_crossing, per_step, per_track = 900.0, 150.0 if case["field"] == "uniform" else 500.0, 330.0
    if case["smoother"] == "two_filter":
        per_crossing, per_step, per_track = 1400.0, 2 * per_step, 1800.0
    flops = n * per_track + (m - n) * (per_crossing + 1.7 * per_step)
    size = 44.0 * m + n * (4 + 160 + 168 + 8 + 8)
    if case["states"]:
        size, flops = size + 160.0 * m, flops + 900.0 * m
    return {"bytes": size, "flops": flops}
