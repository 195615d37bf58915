"""The work that users of this package have it do, as measured cases.

A case names one call pattern (`kind`), a grid, a precision and the number of
time steps of one pass.  Everything goes through the public entry points:
``agcm.Grid``, ``agcm.State``, ``autograd.run`` and ``ensemble.Ensemble``.

    step       State.step(nsteps) and State.store: a forecast
    split      State.step_split: long steps, adaptation in sub-steps
    start      State.load, State.filter, State.diagnostics and State.store: an
               analysis made ready for a run, with its conservation record
    tendency   State.load and State.tendency: the right-hand side for a
               caller's own time integrator
    adjoint    State.step_adjoint: one reverse step of a variational analysis
    gradient   autograd.run and backward: the gradient of a many-step forecast
    ensemble   Ensemble.step and every member's store: members of uneven size

The inputs are a mid-latitude jet with seeded grid-scale noise over seeded
mountains, the kind of state the package's own configurations use, laid out on
the GPU in the state's type.  `exact` states the scheme once more in plain
torch, in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2103_10114_gb300 import agcm, autograd
from paper_2103_10114_gb300.ensemble import Ensemble

FIELDS = ("U", "V", "Phi", "pi")
A_EARTH, OMEGA, R_DRY, C_P, GRAV = 6.371e6, 7.292e-5, 287.04, 1004.64, 9.80665
# the lapse-rate atmosphere with every thermodynamic switch on
THERMO = dict(profile=1, T0=250.0, Ts0=288.15, lapse=6.5e-3, Ttrop=216.65, delta=0.5, delta_c=0.1, delta_p=0.05)
SPLIT = 4       # adaptation sub-steps of a split step
SNAPSHOTS = 3   # stored states of a gradient
MIX = "256x128x30*8,360x180x30*6,720x360x30*2"


def listed():
    def case(name, kind, nlon, nlat, nlev, bits=32, nsteps=1, thermo=False, **more):
        return dict(name=name, kind=kind, nlon=nlon, nlat=nlat, nlev=nlev, bits=bits, nsteps=nsteps, thermo=thermo,
                    **more)

    return [
        # the validation run: a small grid in 64 bits, twenty steps a call; launches and latency count
        case("step-f64-128x64x8", "step", 128, 64, 8, bits=64, nsteps=20),
        # the precision comparison's grid, a usual climate resolution; the state stays in L2
        case("step-f32-256x128x30", "step", 256, 128, 30, nsteps=4),
        # a regional group's own grid: odd counts, rows that are not 16-byte aligned
        case("step-f32-405x203x26", "step", 405, 203, 26, nsteps=2),
        # half a degree and a quarter of a degree, the production resolutions
        case("step-f32-720x360x30", "step", 720, 360, 30, nsteps=2),
        case("step-f32-1440x720x30", "step", 1440, 720, 30, nsteps=2),
        # the 64-bit reference run at half a degree
        case("step-f64-720x360x30", "step", 720, 360, 30, bits=64, nsteps=1),
        # split time stepping, with the lapse-rate atmosphere and the nonlinear term
        case("split-f32-720x360x30", "split", 720, 360, 30, thermo=True),
        # a run's start at a quarter of a degree: load, low-latitude filters, conservation record
        case("start-f32-1440x720x30", "start", 1440, 720, 30),
        # the right-hand side alone, in a caller's own integrator
        case("tendency-f32-512x256x26", "tendency", 512, 256, 26, thermo=True),
        # one reverse step of the half-degree variational problem
        case("adjoint-f32-720x360x30", "adjoint", 720, 360, 30),
        # a whole gradient on the climate grid: forward, recomputation, reverse
        case("gradient-f32-256x128x30", "gradient", 256, 128, 30, nsteps=6),
        # a quarter of the 64-member ensemble's mix, side by side on eight streams
        dict(name="ensemble-f32-mix", kind="ensemble", members=MIX, bits=32, nsteps=2, streams=8),
    ]


def draw(rng):
    most = {32: max(work(c)["bytes"] for c in listed() if c["bits"] == 32),
            64: max(work(c)["bytes"] for c in listed() if c["bits"] == 64)}
    while True:
        case = _any(rng)
        # a reverse step takes as long as three forward ones, and more in 64 bits
        if work(case)["bytes"] * (3 if case["kind"] == "adjoint" and case["bits"] == 64 else 1) <= most[case["bits"]]:
            return case


def _any(rng):
    kind = rng.choice(["step", "step", "step", "step", "split", "start", "tendency", "adjoint", "gradient", "ensemble"])
    bits = 64 if kind in ("step", "adjoint") and rng.random() < 0.3 else 32
    if kind == "ensemble":
        parts = []
        for _ in range(rng.randint(2, 4)):
            nlon = 4 * int(round(math.exp(rng.uniform(math.log(24), math.log(180)))))
            parts.append("%dx%dx%d*%d" % (nlon, nlon // 2 + rng.randint(-2, 2), rng.randint(16, 32), rng.randint(1, 4)))
        return dict(kind=kind, members=",".join(parts), bits=32, nsteps=rng.randint(1, 2), streams=rng.choice([4, 8]))
    # longitudes over the whole range; half of the grids with rows of any length
    hi = 1440 if bits == 32 and kind in ("step", "start", "tendency") else (720 if kind != "gradient" else 360)
    nlon = int(round(math.exp(rng.uniform(math.log(64), math.log(hi)))))
    if rng.random() < 0.5:
        nlon = max(64, nlon // 4 * 4)
    nlat = max(24, int(nlon * rng.uniform(0.4, 0.52)))
    nlev = rng.randint(5, 30)
    nsteps = {"step": rng.randint(1, 2) if nlon > 400 else rng.randint(1, 8), "gradient": rng.randint(3, 6)}.get(kind, 1)
    if bits == 64:
        nsteps = 1 if nlon > 200 else nsteps
    thermo = kind in ("step", "split", "tendency", "adjoint") and rng.random() < 0.3
    return dict(kind=kind, nlon=nlon, nlat=nlat, nlev=nlev, bits=bits, nsteps=nsteps, thermo=thermo)


def _members(case):
    """(nlon, nlat, nlev) of every grid of a case."""
    if case["kind"] != "ensemble":
        return [(case["nlon"], case["nlat"], case["nlev"])]
    out = []
    for part in case["members"].split(","):
        shape, n = part.split("*")
        out += [tuple(int(v) for v in shape.split("x"))] * int(n)
    return out


def _dt(nlon, nlat):
    """A round step below the gravity-wave bound: 30 s at 1440 x 720."""
    return min(43200.0 / nlon, 21600.0 / nlat)


def _inputs(nlon, nlat, nlev, bits, seed):
    """Jet, noise and mountains in the state's type: ({field: tensor}, surface geopotential in 64 bits)."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    f64 = dict(device="cuda", dtype=torch.float64)

    def noise(scale, *shape):
        return scale * torch.randn(*shape, generator=gen, **f64)

    lat = math.pi / 2 - (torch.arange(nlat, **f64) + 0.5) * (math.pi / nlat)
    lon = torch.arange(nlon, **f64) * (2 * math.pi / nlon)
    sig = (torch.arange(nlev, **f64) + 0.5) / nlev
    jet = torch.exp(-(((torch.rad2deg(lat).abs() - 45.0) / 10.0) ** 2))
    prof = torch.exp(-(((sig - 0.25) / 0.3) ** 2))
    U = 35.0 * prof[:, None, None] * jet[None, :, None] + noise(0.35, nlev, nlat, nlon)
    V = noise(0.35, nlev, nlat - 1, nlon)
    Phi = noise(5.0, nlev, nlat, nlon)
    pi = noise(1e-2, nlat, nlon)
    # twelve round mountains of up to 3 km, on the 64-bit grid points
    u = torch.rand(12, 4, generator=gen, **f64)
    height = torch.zeros(nlat, nlon, **f64)
    for a, b, c, d in u.tolist():
        lat0, lon0, w = math.pi * (a - 0.5), 2 * math.pi * b, 0.15 + 0.3 * c
        cosd = math.sin(lat0) * torch.sin(lat)[:, None] + math.cos(lat0) * torch.cos(lat)[:, None] * torch.cos(lon - lon0)
        height = torch.maximum(height, 3000.0 * d * torch.exp((cosd - 1.0) / (w * w)))
    dtype = torch.float64 if bits == 64 else torch.float32
    return {"U": U.to(dtype), "V": V.to(dtype), "Phi": Phi.to(dtype), "pi": pi.to(dtype)}, GRAV * height


def _cotangent(nlon, nlat, nlev, bits, seed):
    """The gradient of a weighted final state: unit noise on every field."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 1_000_003)
    dtype = torch.float64 if bits == 64 else torch.float32
    shapes = {"U": (nlev, nlat, nlon), "V": (nlev, nlat - 1, nlon), "Phi": (nlev, nlat, nlon), "pi": (nlat, nlon)}
    return {f: torch.randn(*s, generator=gen, device="cuda", dtype=torch.float64).to(dtype) for f, s in shapes.items()}


def prepare(case, seed):
    bits, kind = case["bits"], case["kind"]
    states, dts, first = [], [], None
    for n, (nlon, nlat, nlev) in enumerate(_members(case)):
        x, phis = _inputs(nlon, nlat, nlev, bits, seed * 1000 + n)
        grid = agcm.Grid(nlon, nlat, nlev, phis=phis.cpu().numpy(), thermo=THERMO if case.get("thermo") else None)
        s = agcm.State(grid, agcm.AGCM_FP64 if bits == 64 else agcm.AGCM_FP32)
        s.load(x)
        states.append(s)
        dts.append(_dt(nlon, nlat) * (4 if kind == "split" else 1))
        first = first or x
    hold = {"case": case, "s": states[0], "dt": dts[0], "x": first}
    if kind in ("adjoint", "gradient"):
        hold["lam"] = _cotangent(case["nlon"], case["nlat"], case["nlev"], bits, seed)
    if kind == "gradient":
        hold["x"] = {f: v.requires_grad_() for f, v in first.items()}
    if kind == "ensemble":
        hold.update(states=states, dts=dts, ens=Ensemble(states))
        hold["ens"].configure("streams-row", case["streams"])
    torch.cuda.synchronize()
    return hold


def run(state):
    case, s, dt = state["case"], state["s"], state["dt"]
    kind, n = case["kind"], case["nsteps"]
    if kind == "step":
        s.step(n, dt)
        return s.store()
    if kind == "split":
        s.step_split(n, dt, SPLIT)
        return s.store()
    if kind == "start":
        s.load(state["x"])
        s.filter()
        record = s.diagnostics()
        return {**s.store(), **record}
    if kind == "tendency":
        s.load(state["x"])
        return s.tendency()
    if kind == "adjoint":
        return s.step_adjoint(state["lam"], dt)
    if kind == "gradient":
        x, lam = state["x"], state["lam"]
        out = autograd.run(s, x, n, dt, SNAPSHOTS)
        g = torch.autograd.grad([out[f] for f in FIELDS], [x[f] for f in FIELDS], [lam[f] for f in FIELDS])
        return {**{f: v.detach() for f, v in out.items()}, **{"d" + f: v for f, v in zip(FIELDS, g)}}
    state["ens"].step(n, state["dts"])
    return [m.store() for m in state["states"]]


def work(case):
    """A stage of the three-stage step depends on whole columns and on
    neighbours of the stage before, so each stage reads its input (and, after
    the first, the step's start) and writes its output: 24 words a point and
    step.  163 operations a point and stage is the scheme's own count."""
    word = case["bits"] // 8
    pts = sum(i * j * k for i, j, k in _members(case))
    kind, n = case["kind"], case["nsteps"]
    words, stages = 24, 3
    if kind == "split":
        words, stages = 24 * (SPLIT + 1), 1.5 * (SPLIT + 1)   # half of the terms in each
    elif kind == "start":
        words, stages = 6 + 6 + 3 + 6, 0.1                    # load, filter in place, one reading for the sums, store
    elif kind == "tendency":
        words, stages = 6 + 6, 1                              # load, then fields in and tendency out
    elif kind == "adjoint":
        words, stages = 15 + 3 * 9 + 12, 2 + 3 * 2            # two stages again, three products, sums
    elif kind == "gradient":
        words, stages = 24 + 54, 3 + 8
    if kind in ("step", "split", "ensemble"):
        words += 6 / n                                        # the store
    return {"bytes": words * word * pts * n, "flops": 163 * stages * pts * n}


# ---------------------------------------------------------------------------
# The scheme in plain torch, in 64 bits.


def _stride(theta, dlam):
    r = math.asin(math.sqrt(0.5) * math.sin(dlam)) / math.asin(math.sin(theta) * math.sin(dlam))
    n = max(1, math.ceil(r - 1e-9))
    return n if n % 2 else n + 1


class _Scheme:
    def __init__(self, nlon, nlat, nlev, phis, thermo):
        def row(v):
            return torch.tensor(v, dtype=torch.float64, device="cuda")[:, None]

        I, J, K = nlon, nlat, nlev
        self.I, self.J, self.K = I, J, K
        self.dlam, self.dth = 2 * math.pi / I, math.pi / J
        ths, thv = [(j + 0.5) * self.dth for j in range(J)], [(j + 1.0) * self.dth for j in range(J - 1)]
        self.s, self.sv = row([math.sin(t) for t in ths]), row([math.sin(t) for t in thv])
        self.f0 = 2 * OMEGA * row([math.cos(t) for t in ths])
        self.cot = row([math.cos(t) / math.sin(t) for t in ths]) / A_EARTH
        self.area = A_EARTH ** 2 * self.dth * self.dlam * self.s
        self.areav = A_EARTH ** 2 * self.dth * self.dlam * self.sv
        self.lat, self.latv = [90.0 - t * 180.0 / math.pi for t in ths], [90.0 - t * 180.0 / math.pi for t in thv]
        self.M, self.Mv = [_stride(t, self.dlam) for t in ths], [_stride(t, self.dlam) for t in thv]
        self.Mr, self.Mvr = row([float(m) for m in self.M]), row([float(m) for m in self.Mv])
        sh = np.arange(K + 1) / K
        mid, H = 0.5 * (sh[1:] + sh[:-1]), np.zeros((K, K))
        for k in range(K):
            H[k, k] = math.log(sh[k + 1] / mid[k])
            for q in range(k + 1, K):
                H[k, q] = math.log(sh[q + 1] / sh[q])
        self.H = torch.tensor(H, device="cuda")
        self.sh = torch.tensor(sh, device="cuda")[:, None, None]
        self.ds = 1.0 / K
        t = thermo
        if t is None:
            temp, pit, ts = np.full(K, 250.0), torch.exp(-phis / (R_DRY * 250.0)), torch.full_like(phis, 250.0)
            t = dict(delta=0.0, delta_c=0.0, delta_p=0.0)
        else:
            temp = np.maximum(t["Ts0"] * mid ** (R_DRY * t["lapse"] / GRAV), t["Ttrop"])
            ts = torch.clamp(t["Ts0"] - t["lapse"] / GRAV * phis, min=t["Ttrop"])
            above = torch.clamp(phis / GRAV - (t["Ts0"] - t["Ttrop"]) / t["lapse"], min=0.0)
            pit = (ts / t["Ts0"]) ** (GRAV / (R_DRY * t["lapse"])) * torch.exp(-GRAV * above / (R_DRY * t["Ttrop"]))
        kap = R_DRY / C_P
        beta = (1 - t["delta_p"]) * (1 + t["delta_c"]) * np.sqrt(kap * R_DRY * temp)
        self.beta = torch.tensor(beta, device="cuda")[:, None, None]
        self.beta2 = (1 - t["delta_p"]) * t["delta"] * kap
        self.pit, self.surf = pit, R_DRY * ts / pit

    def at(self, F, offs):
        """F at longitude index i + offs[j] of every row j."""
        idx = torch.arange(self.I, device="cuda")[None, :] + torch.tensor(offs, device="cuda")[:, None]
        return F.gather(-1, (idx % self.I).expand(F.shape))

    def tendency(self, x, adv=True, ada=True):
        U, V, Phi, pi = x
        a, K, M, Mv = A_EARTH, self.K, self.M, self.Mv
        lo, hi = [(m - 1) // 2 for m in M], [(m + 1) // 2 for m in M]
        neg = lambda v: [-q for q in v]
        east, west = lambda F: F.roll(-1, -1), lambda F: F.roll(1, -1)
        rows = lambda F: torch.nn.functional.pad(F, (0, 0, 1, 1))   # V rows with the pole edges, where V is zero
        m = self.pit + pi
        P, Pu, Pv = m.sqrt(), (0.5 * (m + east(m))).sqrt(), (0.5 * (m[:-1] + m[1:])).sqrt()
        Fl, Ft = Pu * U, Pv * V
        dx, dy = a * self.s * self.Mr * self.dlam, a * self.s * self.dth
        FlE, FlW = self.at(Fl, lo), self.at(Fl, neg(hi))
        q = rows(self.sv * Ft)
        D = (FlE - FlW) / dx + (q[:, 1:] - q[:, :-1]) / dy
        C = self.ds * D.sum(0)
        tU, tV, tPhi, tpi = torch.zeros_like(U), torch.zeros_like(V), torch.zeros_like(Phi), torch.zeros_like(pi)
        if ada:
            c = (self.beta + self.beta2 * Phi / P) / P
            psi = (self.H @ (c * Phi).reshape(K, -1)).reshape(Phi.shape) + self.surf * pi
            tU = tU - Pu * (self.at(psi, hi) - self.at(psi, neg(lo))) / dx
            tV = tV - Pv * (psi[:, 1:] - psi[:, :-1]) / (a * self.dth)
            tPhi = tPhi - c * (self.H.T @ D.reshape(K, -1)).reshape(D.shape)
            fU = (self.f0 + U / Pu * self.cot)
            v = rows(V + east(V))
            tU = tU - 0.25 * fU * (v[:, 1:] + v[:, :-1])
            g = self.area * fU * U
            g = g + west(g)
            tV = tV + 0.25 * (g[:, 1:] + g[:, :-1]) / self.areav
            tpi = -C
        if adv:
            W = torch.cat([torch.zeros_like(D[:1]), self.sh[1:K] * C - self.ds * D.cumsum(0)[:-1], torch.zeros_like(D[:1])])
            Gs, Gu, Gv = Phi / P, U / Pu, V / Pv
            updown = lambda w, G: (torch.nn.functional.pad(w[1:K] * G[1:], (0, 0, 0, 0, 0, 1))
                                   - torch.nn.functional.pad(w[1:K] * G[:-1], (0, 0, 0, 0, 1, 0))) / (2 * self.ds)
            nb = lambda G: (rows(G)[:, 2:], rows(G)[:, :-2])        # rows j+1 and j-1
            zf, zfv = a * self.dth / self.Mr, a * self.dth / self.Mvr
            y = rows(a * self.dlam * self.sv * Ft)
            yS, yN = y[:, 1:], y[:, :-1]
            S, N = nb(Gs)
            hor = zf * (FlE * self.at(Gs, M) - FlW * self.at(Gs, neg(M))) + yS * S - yN * N
            tPhi = tPhi - (hor / (2 * self.area) + updown(W, Gs)) / P
            S, N = nb(Gu)
            ZE, ZW = 0.5 * zf * (FlE + self.at(Fl, hi)), 0.5 * zf * (FlW + self.at(Fl, neg(lo)))
            hor = ZE * self.at(Gu, M) - ZW * self.at(Gu, neg(M)) + 0.5 * ((yS + east(yS)) * S - (yN + east(yN)) * N)
            tU = tU - (hor / (2 * self.area) + updown(0.5 * (W + east(W)), Gu)) / Pu
            S, N = nb(Gv)
            lov, hiv = [(v - 1) // 2 for v in Mv], [(v + 1) // 2 for v in Mv]
            Fm = 0.5 * zfv
            ZE = Fm * (self.at(Fl[:, :-1], lov) + self.at(Fl[:, 1:], lov))
            ZW = Fm * (self.at(Fl[:, :-1], neg(hiv)) + self.at(Fl[:, 1:], neg(hiv)))
            yv = a * self.dlam * self.sv * Ft
            S2, N2 = nb(yv)
            hor = ZE * self.at(Gv, Mv) - ZW * self.at(Gv, neg(Mv)) + 0.5 * ((yv + S2) * S - (yv + N2) * N)
            tV = tV - (hor / (2 * self.areav) + updown(0.5 * (W[:, :-1] + W[:, 1:]), Gv)) / Pv
        return tU, tV, tPhi, tpi

    def step(self, x, dt, **terms):
        y = x
        for c in (0.5, 0.5, 1.0):
            y = tuple(b + c * dt * t for b, t in zip(x, self.tendency(y, **terms)))
        return y

    def vjp(self, x, lam, dt):
        x = tuple(v.detach().requires_grad_() for v in x)
        with torch.enable_grad():
            return torch.autograd.grad(self.step(x, dt), x, lam)

    def filtered(self, x):
        sign = torch.ones(self.I, dtype=torch.float64, device="cuda")
        sign[1::2] = -1.0

        def one(F, lat):
            lat = torch.tensor(lat, dtype=torch.float64, device="cuda").abs()[:, None]
            G = F + 0.25 * (F.roll(1, -1) - 2 * F + F.roll(-1, -1))
            wave = sign * (sign * F).mean(-1, keepdim=True) if self.I % 2 == 0 else torch.zeros_like(F)
            return torch.where(lat < 38.0, F - wave, torch.where(lat <= 70.0, G, F))

        return tuple(one(F, self.latv if n == 1 else self.lat) for n, F in enumerate(x))

    def record(self, x):
        U, V, Phi, pi = x
        kin = 0.5 * self.ds * ((self.area * U * U).sum() + (self.areav * V * V).sum())
        pot, ps = 0.5 * self.ds * (self.area * Phi * Phi).sum(), 0.5 * (self.area * self.surf * pi * pi).sum()
        v = {"mass": (self.area * (self.pit + pi)).sum(), "e_kin": kin, "e_pot": pot, "e_ps": ps,
             "energy": kin + pot + ps, "max_u": U.abs().max(), "max_v": V.abs().max()}
        return {**{k: float(t) for k, t in v.items()}, "finite": 1}


def exact(case, seed):
    kind, n, out = case["kind"], case["nsteps"], []
    with torch.no_grad():
        for q, (nlon, nlat, nlev) in enumerate(_members(case)):
            first, phis = _inputs(nlon, nlat, nlev, case["bits"], seed * 1000 + q)
            x = tuple(first[f].double() for f in FIELDS)
            sch = _Scheme(nlon, nlat, nlev, phis, THERMO if case.get("thermo") else None)
            dt = _dt(nlon, nlat)
            if kind == "tendency":
                return dict(zip(FIELDS, sch.tendency(x)))
            if kind == "start":
                x = sch.filtered(x)
                return {**dict(zip(FIELDS, x)), **sch.record(x)}
            if kind in ("adjoint", "gradient"):
                lam = _cotangent(nlon, nlat, nlev, case["bits"], seed)
                g, xs = tuple(lam[f].double() for f in FIELDS), [x]
                if kind == "adjoint":
                    return dict(zip(FIELDS, sch.vjp(x, g, dt)))
                for _ in range(n):
                    xs.append(sch.step(xs[-1], dt))
                for y in reversed(xs[:-1]):
                    g = sch.vjp(y, g, dt)
                return {**dict(zip(FIELDS, xs[-1])), **{"d" + f: v for f, v in zip(FIELDS, g)}}
            for _ in range(n):
                if kind == "split":
                    for _ in range(SPLIT):
                        x = sch.step(x, 4 * dt / SPLIT, adv=False)
                    x = sch.step(x, 4 * dt, ada=False)
                else:
                    x = sch.step(x, dt)
            out.append(dict(zip(FIELDS, x)))
    return out if kind == "ensemble" else out[0]
