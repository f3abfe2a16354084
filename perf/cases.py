"""Performance cases of the active lattice Boltzmann library.

Each case is work a user of the library has it do through `Simulation` and
`regimes.density_sweep`: advancing single lattices and batches and reading the
populations back, the paper's density sweep, exchanging fields on the device
and with the host.  `exact` restates the method in 64-bit torch, from the
paper and from the conventions that `include/lbm.h` documents (lattices,
random numbers, initial states, storage shifts), without the package.

A case's fields: `kind` ("advance", "sweep", "fields", "host"); `q` (9: D2Q9,
7: the paper's D2Q7); `nx`, `ny`, `n` (lattices of one size), or `sides` and
`mix` (the sizes a ragged batch draws from, and the seed of the drawing);
`model`; `storage`; `scale` ("rho1": parameters at mean density 1, "paper":
the paper's own numbers); `start` ("random", or "ordered" along x); `steps` (of
one pass; of one sweep point); `every` (sampling interval, 0: none).
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_1902_00530_gb300 import Lattice, Simulation
from paper_1902_00530_gb300.regimes import density_sweep

RATE = {"f32": 4, "f16s": 2, "bf16s": 2}  # bytes of a stored population
KEYS = ("t", "mass", "phi", "drho_y", "drho_x", "var_rho", "zeta")


def _case(name, kind="advance", q=9, nx=0, ny=0, n=1, model="cil", storage="f32", scale="rho1", start="random",
          steps=1, every=0, sides="", mix=0):
    c = dict(kind=kind, q=q, nx=nx, ny=ny, n=n, model=model, storage=storage, scale=scale, start=start, steps=steps,
             every=every, sides=sides, mix=mix)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's phase-diagram box of the MIPS model, one run at a high noise: a short
        # relaxation, then the state; the smallest lattice in use, bound by latency and launches
        _case("mips7_90x30", q=7, nx=90, ny=30, model="mips", scale="paper", steps=100),
        # a few steps of a 64 x 64 lattice, as in a parity check or an interactive look
        _case("mips9_64_short", nx=64, ny=64, model="mips", steps=10),
        # the paper's hysteresis procedure: 32 boxes of 180 x 60 as one batch, one density point
        # up and one down, every lattice sampled at both
        _case("sweep7_32x180x60", kind="sweep", q=7, nx=180, ny=60, n=32, scale="paper", start="ordered", steps=500),
        # the paper's critical snapshot box, 720 x 240
        _case("cil7_720x240", q=7, nx=720, ny=240, scale="paper", steps=100),
        # a 1024 x 1024 run with its observables sampled every 100 steps; lives in the L2 cache
        _case("cil9_1024_sampled", nx=1024, ny=1024, steps=100, every=100),
        # sides that no vector width divides, 16-bit storage, no noise
        _case("passive9_1021x777_bf16", nx=1021, ny=777, model="passive", storage="bf16s", steps=50),
        # the large single lattice with noise
        _case("mips9_8192", nx=8192, ny=8192, model="mips", steps=20),
        # a large box of the paper's own lattice
        _case("mips7_4096", q=7, nx=4096, ny=4096, model="mips", steps=20),
        # the batch over a density x activity grid
        _case("cil9_batch_256x256x256", nx=256, ny=256, n=256, steps=50),
        # lattices of several sizes and both closures in one 16-bit batch
        _case("mixed9_ragged_64_bf16", n=64, model="mixed", storage="bf16s", steps=10,
              sides="128,256,512,1024,2048", mix=190200535),
        # reading and restoring a state on the device: moments, observables, populations out and in
        _case("fields9_4096_bf16", kind="fields", nx=4096, ny=4096, model="mips", storage="bf16s"),
        # offloading a 16-bit state to pinned host memory and bringing it back
        _case("host9_1024_f16", kind="host", nx=1024, ny=1024, model="cil", storage="f16s"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["advance"] * 6 + ["sweep", "fields", "host"])
    q = rng.choice([9, 9, 7])
    model = rng.choice(["mips", "cil", "passive"])
    storage = rng.choice(["f32", "f32", "f16s", "bf16s"])
    scale = rng.choice(["rho1", "paper"]) if q == 7 and model != "passive" else "rho1"
    if kind == "sweep":
        n = _log(rng, 2, 48)
        nx, ny = _log(rng, 60, 360), 2 * _log(rng, 15, 80)
        return _case("", kind, 7, nx, ny, n, "cil", rng.choice(["f32", "f16s"]), "paper", "ordered", _log(rng, 50, 500))
    nx, ny = _log(rng, 24, 4096), _log(rng, 24, 4096)
    if rng.random() < 0.5:
        nx = max(32, nx // 32 * 32)
    if q == 7:
        ny += ny % 2
    if kind in ("fields", "host"):
        ny = min(ny, (1 << (24 if kind == "fields" else 21)) // nx // 2 * 2)
        return _case("", kind, q, nx, ny, 1, model, storage, scale)
    n = rng.choice([1, 1, 1, _log(rng, 2, 64)])
    steps = _log(rng, 2, 100)
    while n * nx * ny * steps > 3e8:
        if steps > 8:
            steps //= 2
        elif n > 1:
            n //= 2
        else:
            ny = ny // 4 * 2
    return _case("", kind, q, nx, ny, n, model, storage, scale, rng.choice(["random", "ordered"]), steps,
                 rng.choice([0, 0, max(1, steps // 3)]))


# ------------------------------------------------------------------ parameters
def _params(case, model, k, n):
    """(parameters, initial state) of lattice k of n: the paper's numbers (App.
    C.1, C.2; on D2Q9 sigma / sqrt 2), or their images at mean density 1; a
    batch spreads over mean density and activity."""
    paper = case["scale"] == "paper"
    noise = 1.0 if case["q"] == 7 else math.sqrt(0.5)
    spec = dict(rho_mean=1.0, rho_amp=0.01, u_kind=0, u_amp=1e-3, ux0=0.0, uy0=0.0)
    if model == "mips":
        rho = 0.12
        p = dict(tau=2.0 if case["q"] == 7 else 1.0, sigma=(3.0 / 70.0 if paper else 0.014) * noise, C=50.0,
                 rho_star=0.2, u_max=0.3)
    elif model == "cil":
        rho = 0.185
        p = dict(tau=1.0, sigma=noise / 70.0, A=2.0, B=0.3)
        if n > 1 and case["kind"] == "advance":
            p["B"] = 0.3 * (0.25 + 0.75 * (k % 16) / 15.0)
        if case["start"] == "ordered":
            spec["ux0"] = max(p["B"] - p["A"] * rho * rho, 0.0)
        else:
            spec.update(rho_amp=0.1, u_kind=1, u_amp=0.01)
    else:
        rho, p = 1.0, dict(tau=1.0)
        spec.update(rho_amp=0.1, u_kind=1, u_amp=0.01)
    if paper:
        spec["rho_mean"] = rho
    else:  # the density-rescaling image at mean density 1
        for key, f in (("sigma", 1.0 / rho), ("C", rho), ("rho_star", 1.0 / rho), ("A", rho * rho)):
            if key in p:
                p[key] *= f
    if n > 1 and case["kind"] == "advance":
        spec["rho_mean"] *= 0.7 + 0.6 * (k // 16) / max(1, (n - 1) // 16)
    return p, spec


def _lattices(case):
    """[(nx, ny, model)] of the case."""
    if case["sides"]:
        r = random.Random(case["mix"])
        sides = [int(s) for s in case["sides"].split(",")]
        return [(s, s, r.choice(["mips", "cil"])) for s in (r.choice(sides) for _ in range(case["n"]))]
    return [(case["nx"], case["ny"], case["model"])] * case["n"]


DELTA = 0.0025  # the density step of the paper's sweeps


# ---------------------------------------------------------------- the program
def prepare(case, seed):
    lats = _lattices(case)
    ps = [_params(case, m, k, len(lats)) for k, (_, _, m) in enumerate(lats)]
    vs = "d2q7" if case["q"] == 7 else "d2q9"
    sim = Simulation([Lattice(x, y, case["storage"], k, vs) for k, (x, y, _) in enumerate(lats)],
                     [m for _, _, m in lats], [p for p, _ in ps], sample_every=case["every"],
                     ring_capacity=64 if case["every"] else 0)
    sim.init(seed, [s for _, s in ps])
    if case["kind"] in ("advance", "sweep"):
        sim.tune()
    q = case["q"]
    total = sum(q * x * y for x, y, _ in lats)
    f = torch.empty(total, dtype=torch.float32, pin_memory=True) if case["kind"] == "host" else \
        torch.empty(total, dtype=torch.float32, device="cuda")
    views, at = [], 0
    for x, y, _ in lats:
        views.append(f[at:at + q * x * y].view(q, y, x))
        at += q * x * y
    return dict(case=case, sim=sim, f=f, views=views, rho=ps[0][1]["rho_mean"])


def _rows(records):
    return torch.tensor([[r[k] for k in KEYS] for r in records], dtype=torch.float64)


def run(state):
    case, sim = state["case"], state["sim"]
    if case["kind"] == "advance":
        sim.step(case["steps"])
        out = {}
        if case["every"]:
            out["series"] = [_rows(sim.observable_series(k, cap=64)) for k in range(min(case["n"], 32))]
        for k, v in enumerate(state["views"]):
            sim.get_state(k, out=v)
        return dict(out, f=state["f"])
    if case["kind"] == "sweep":
        rho, every = state["rho"], list(range(case["n"]))
        up = density_sweep(sim, rho, rho, DELTA, case["steps"], sample=every)
        down = density_sweep(sim, rho + DELTA, rho + DELTA, -DELTA, case["steps"], sample=every)
        for k, v in enumerate(state["views"]):
            sim.get_state(k, out=v)
        return dict(up=_rows(up[0][1]), down=_rows(down[0][1]), f=state["f"])
    if case["kind"] == "fields":
        rho, ux, uy = sim.moments()
        obs = _rows([sim.observables()])
        sim.get_state(out=state["views"][0])
        sim.set_state(state["views"][0])
        return dict(rho=rho, ux=ux, uy=uy, obs=obs, f=state["f"])
    sim.get_state(out=state["views"][0])
    sim.set_state(state["views"][0])
    return dict(f=state["f"])


def work(case):
    q, e, model = case["q"], RATE[case["storage"]], case["model"]
    sites = sum(x * y for x, y, _ in _lattices(case))
    if case["kind"] == "fields":  # read the stored state for moments, observables, populations out; write both ways
        return dict(bytes=sites * (3 * q * e + 12 + q * 4 + q * 4 + q * e), flops=sites * 60)
    if case["kind"] == "host":
        return dict(bytes=sites * 2 * q * (e + 4), flops=0)
    steps = case["steps"] * (2 if case["kind"] == "sweep" else 1)
    # an update reads and writes each population once, and does about this many floating operations
    per = {9: 130, 7: 100}[q] + (0 if model == "passive" else 20) + (30 if model in ("mips", "mixed") else 0)
    return dict(bytes=sites * (2 * q * e * steps + q * (e + 4)), flops=sites * steps * per)


# ------------------------------------------------- the method in 64-bit torch
M0, M1, K0, K1, U32 = 0xD2511F53, 0xCD9E8D57, 0x9E3779B9, 0xBB67AE85, 0xFFFFFFFF
E9 = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
E7 = [(0, 0), (2, 0), (1, 1), (-1, 1), (-2, 0), (-1, -1), (1, -1)]  # (2 e_x, row offset)
W9 = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
W7 = [1 / 2] + [1 / 12] * 6
H3 = math.sqrt(3.0) / 2


def _philox(c, key):
    """Philox4x32-10 of four int64 tensors of 32-bit words."""
    x, y, z, w = c
    k0, k1 = key & U32, (key >> 32) & U32
    for r in range(10):
        p0, p1 = x * M0, z * M1  # wrap modulo 2^64: the halves are taken by masks
        x, y, z, w = (((p1 >> 32) & U32) ^ y ^ ((k0 + r * K0) & U32), p1 & U32,
                      ((p0 >> 32) & U32) ^ w ^ ((k1 + r * K1) & U32), p0 & U32)
    return x, y, z, w


def _counter(g, t, word):
    return (g["x"].expand(g["shape"]), g["y"].expand(g["shape"]),
            torch.full(g["shape"], t, dtype=torch.int64, device="cuda"), (g["id"] | word).expand(g["shape"]))


def _e(q, i):
    return E9[i] if q == 9 else (E7[i][0] / 2, E7[i][1] * H3)


def _from(a, q, i, s):
    """a at r + s e_i, for every site r (a: [lattice, y, x])."""
    dx, dy = (s * v for v in (E9 if q == 9 else E7)[i])
    if q == 9:
        return torch.roll(a, (-dy, -dx), (1, 2))
    out = torch.empty_like(a)
    b = torch.roll(a, -dy, 1)
    for par in (0, 1):  # site (x, y) sits at x + (y mod 2) / 2
        shift = (dx + par - (par + dy) % 2) // 2
        out[:, par::2] = torch.roll(b[:, par::2], -shift, 2)
    return out


def _equilibrium(q, rho, ux, uy):
    a, b, c = (3.0, 4.5, 1.5) if q == 9 else (4.0, 8.0, 2.0)
    u2 = ux * ux + uy * uy
    out = []
    for i, w in enumerate(W9 if q == 9 else W7):
        ex, ey = _e(q, i)
        eu = ex * ux + ey * uy
        out.append(w * rho * (1.0 + a * eu + b * eu * eu - c * u2))
    return out


def _col(g, name):
    return torch.tensor([p.get(name, 0.0) for p, _ in g["ps"]], dtype=torch.float64, device="cuda").view(-1, 1, 1)


def _spec(g, name):
    return torch.tensor([float(s[name]) for _, s in g["ps"]], dtype=torch.float64, device="cuda").view(-1, 1, 1)


def _initial(case, g, seed):
    q = case["q"]
    w = _philox(_counter(g, 0, 1 << 24), seed)
    u = [((v >> 8).double() + 0.5) / 16777216.0 for v in w[:3]]
    rho = _spec(g, "rho_mean") * (1.0 + _spec(g, "rho_amp") * (2.0 * u[0] - 1.0))
    amp = _spec(g, "u_amp")
    if g["ps"][0][1]["u_kind"] == 0:
        ux, uy = _spec(g, "ux0") + amp * (2.0 * u[1] - 1.0), _spec(g, "uy0") + amp * (2.0 * u[2] - 1.0)
    else:
        ux = _spec(g, "ux0") + amp * torch.cos(2 * math.pi * u[1])
        uy = _spec(g, "uy0") + amp * torch.sin(2 * math.pi * u[1])
    f = _equilibrium(q, rho, ux, uy)
    kind = {"f32": torch.float32, "f16s": torch.float16, "bf16s": torch.bfloat16}[case["storage"]]
    if kind == torch.float32:
        return [v.float().double() for v in f]
    shift = [(_spec(g, "rho_mean") * v).float().to(kind).double() for v in (W9 if q == 9 else W7)]
    return [(v - s).to(kind).double() + s for v, s in zip(f, shift)]


def _moments(q, f):
    rho = sum(f)
    jx = sum(_e(q, i)[0] * f[i] for i in range(1, q))
    jy = sum(_e(q, i)[1] * f[i] for i in range(1, q))
    return rho, jx, jy


def _step(q, model, g, f, seed, t):
    f = [_from(f[i], q, i, -1) for i in range(q)]
    rho, jx, jy = _moments(q, f)
    if model == "mips":
        nb = [_from(rho, q, i, 1) for i in range(1, q)]
        cs = 3.0 if q == 9 else 4.0
        wt = (W9 if q == 9 else W7)[1:]
        gx = cs * sum(w * _e(q, i + 1)[0] * v for i, (w, v) in enumerate(zip(wt, nb)))
        gy = cs * sum(w * _e(q, i + 1)[1] * v for i, (w, v) in enumerate(zip(wt, nb)))
        c = torch.where(rho < _col(g, "rho_star"), _col(g, "C") * (1.0 - rho / _col(g, "rho_star")), 0.0)
        sx, sy = c * gx, c * gy
        m = torch.sqrt(sx * sx + sy * sy)
        s = torch.where(m > _col(g, "u_max"), _col(g, "u_max") / m, 1.0)
        sx, sy = sx * s, sy * s
    elif model == "cil":
        m = torch.sqrt(jx * jx + jy * jy)
        u0 = torch.clamp(_col(g, "B") - _col(g, "A") * rho * rho, min=0.0)
        s = torch.where((m > 0) & (rho > 0), u0 / m, 0.0)
        sx, sy = jx * s, jy * s
    else:
        s = torch.where(rho > 0, 1.0 / rho, 0.0)
        sx, sy = jx * s, jy * s
    om = 1.0 / _col(g, "tau")
    f = [v + om * (e - v) for v, e in zip(f, _equilibrium(q, rho, sx, sy))]
    if any(p.get("sigma", 0.0) > 0 for p, _ in g["ps"]):
        w = _philox(_counter(g, t, 0), seed)
        if q == 9:
            m = []
            for v in w:
                m += [v >> 18, (v >> 4) & 0x3FFF]
            m.append((w[0] & 15) | (w[1] & 15) << 4 | (w[2] & 15) << 8 | (w[3] & 3) << 12)
            s = [(2 * v + 1 - 16384).double() / 16384.0 for v in m]
        else:
            s = [(2 * ((w[i >> 1] >> 16) if i & 1 else (w[i >> 1] & 0xFFFF)) + 1 - 65536).double() / 65536.0
                 for i in range(7)]
        mean = sum(s) / q
        f = [v + _col(g, "sigma") * (n - mean) for v, n in zip(f, s)]
    bad = f[0] < 0
    f[0] = torch.clamp(f[0], min=0.0)
    for a, b in [(1, 3), (2, 4), (5, 7), (6, 8)] if q == 9 else [(1, 4), (2, 5), (3, 6)]:
        bad = bad | (f[a] < 0) | (f[b] < 0)
        na = torch.clamp(f[a], max=0.0)
        f[a], f[b] = f[a] - na, f[b] - na
        nb = torch.clamp(f[b], max=0.0)
        f[a], f[b] = f[a] - nb, f[b] - nb
    s = torch.where(bad, rho / sum(f), 1.0)
    return [v * s for v in f]


def _observables(q, f, b, t):
    rho, jx, jy = _moments(q, f)
    mass = rho.sum()
    zeta = b - torch.sqrt(jx * jx + jy * jy).sum() / mass
    v = [mass, torch.hypot(jx.sum(), jy.sum()) / mass, rho.mean(0).std(unbiased=False),
         rho.mean(1).std(unbiased=False), rho.var(unbiased=False), zeta]
    return [float(t)] + [float(x) for x in v]


def exact(case, seed):
    """None where the trajectory decorrelates at rounding level within the
    pass: the disordered CIL start, and the long sweeps."""
    steps = case["steps"]
    if case["kind"] == "sweep" and steps > 100 or case["kind"] == "advance" and \
            case["model"] in ("cil", "mixed") and case["start"] == "random" and steps > 60:
        return None
    q, lats = case["q"], _lattices(case)
    ps = [_params(case, m, k, len(lats)) for k, (_, _, m) in enumerate(lats)]
    groups = {}
    for k, key in enumerate(lats):
        groups.setdefault(key, []).append(k)
    flat, series, up, down = [None] * len(lats), {}, {}, {}
    for (nx, ny, model), members in groups.items():
        ids = torch.tensor(members, dtype=torch.int64, device="cuda").view(-1, 1, 1)
        g = dict(ps=[ps[k] for k in members], id=ids, shape=(len(members), ny, nx),
                 x=torch.arange(nx, dtype=torch.int64, device="cuda").view(1, 1, -1),
                 y=torch.arange(ny, dtype=torch.int64, device="cuda").view(1, -1, 1))
        f = _initial(case, g, seed)

        def sample(into, t):
            for j, k in enumerate(members):
                into.setdefault(k, []).append(_observables(q, [v[j] for v in f], ps[k][0].get("B", 0.0), t))

        if case["kind"] == "advance":
            for t in range(steps):
                f = _step(q, model, g, f, seed, t)
                if case["every"] and (t + 1) % case["every"] == 0:
                    sample(series, t + 1)
        elif case["kind"] == "sweep":
            for t in range(2 * steps):
                f = _step(q, model, g, f, seed, t)
                if t + 1 in (steps, 2 * steps):
                    sample(up if t < steps else down, t + 1)
                    f = [v + (DELTA if t < steps else -DELTA) / q for v in f]
        elif case["kind"] == "fields":
            sample(up, 0)
            rho, jx, jy = _moments(q, [v[0] for v in f])
        for j, k in enumerate(members):
            flat[k] = torch.stack([v[j] for v in f]).reshape(-1)
    out = dict(f=torch.cat(flat))
    if case["kind"] == "advance" and case["every"]:
        out["series"] = [torch.tensor(series.get(k, []), dtype=torch.float64).reshape(-1, len(KEYS))
                         for k in range(min(case["n"], 32))]
    if case["kind"] == "sweep":
        out.update(up=torch.tensor([up[k][0] for k in range(len(lats))], dtype=torch.float64),
                   down=torch.tensor([down[k][0] for k in range(len(lats))], dtype=torch.float64))
    if case["kind"] == "fields":
        out.update(rho=rho, ux=jx / rho, uy=jy / rho, obs=torch.tensor(up[0], dtype=torch.float64))
    return out
