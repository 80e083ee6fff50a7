"""Measured cases: what a user of the library has it do, through its public calls.

A case is one of six kinds of work:

  solve     device fields -> f^eq -> n time steps -> moments, one simulation
            (Simulation, dbm_init_state_device, dbm_step, dbm_moments_device)
  host      the same from and to pinned host arrays (dbm_init_state, dbm_moments)
  batch     many uneven simulations advanced together (Batch)
  serve     requests through submit / poll on host arrays (Server)
  noneq     the non-equilibrium manifestations of a state in hand (dbm_noneq_device)
  diagnose  moments and non-equilibrium manifestations of a state in hand

Sizes, rates and shapes follow workloads.py, the benchmark's legs and the tests:
annuli of 64^2 to 2048^2 sites, the pi/4 sectors of one theta cell that the
paper's own runs use (2000 to 24000 radial sites), and sweeps of uneven squares.
exact() restates the update in plain torch FP64.
"""
import math

import numpy as np
import torch

from paper_1308_0653_gb300 import dbm
from paper_1308_0653_gb300 import workloads as W

NV = 33
FIELDS = ("rho", "ur", "uth", "T", "lam")


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _solve(name, shape, nr, ntheta, precision, steps, kind="solve", consistent=False, exponents=False):
    return {"name": name, "kind": kind, "shape": shape, "nr": nr, "ntheta": ntheta, "precision": precision,
            "steps": steps, "consistent": consistent, "exponents": exponents}


def listed():
    return [
        # the small FP64 configuration, whole: 64 x 64, 200 steps; launches count
        _solve("explosion64_fp64", "inert", 64, 64, "fp64", 200),
        # a stretch of the 512 x 512 reactive explosion (its state stays in L2)
        _solve("explosion512_fp32", "explosion", 512, 512, "fp32", 100),
        # the headline benchmark: 2048 x 2048 reactive implosion, 20 steps
        _solve("implosion2048_fp32", "implosion", 2048, 2048, "fp32", 20),
        # the benchmark's FP64 arm on the same grid
        _solve("implosion2048_fp64", "implosion", 2048, 2048, "fp64", 4),
        # the paper's explosion run: a disc of one pi/4 sector cell, FP32
        _solve("sector6000_fp32", "sector", 6000, 1, "fp32", 400),
        # the paper's validation detonation at its own resolution, FP64
        _solve("planar20000_fp64", "planar", 20000, 1, "fp64", 200),
        # odd sizes with the other options: heat from the lambda increment, pow()
        _solve("ragged777x501_fp32", "explosion", 777, 501, "fp32", 50, consistent=True, exponents=True),
        # the end-to-end call: pinned host fields in, 20 steps, host moments out
        _solve("host1024_fp32", "implosion", 1024, 1024, "fp32", 20, kind="host"),
        # a parameter sweep of uneven instances in shared launches
        {"name": "sweep24_fp32", "kind": "batch", "instances": 24, "nmin": 128, "nmax": 640, "precision": "fp32",
         "steps": 96},
        # requests through the server, host arrays both ways
        {"name": "serve8_fp32", "kind": "serve", "instances": 8, "nmin": 128, "nmax": 512, "precision": "fp32",
         "steps": 400},
        # Delta* fields of the FP32 benchmark grid (the paper's Sec. II.E output)
        {"name": "noneq2048_fp32", "kind": "noneq", "nr": 2048, "ntheta": 2048, "precision": "fp32"},
        # all diagnostics of an FP64 state
        {"name": "diagnose1000x900_fp64", "kind": "diagnose", "nr": 1000, "ntheta": 900, "precision": "fp64"},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(("solve", "solve", "solve", "sector", "host", "batch", "serve", "noneq", "diagnose"))
    prec = rng.choice(("fp32", "fp64"))
    if kind == "solve":
        nr, nth = _log(rng, 48, 2048), _log(rng, 48, 2048)
        # a cost bound in site-steps: FP64 arithmetic is some 25 times dearer
        cap = (8e7 if prec == "fp32" else 1e7) / (nr * nth)
        opt = rng.random() < 0.25
        return dict(_solve("", rng.choice(("explosion", "implosion", "inert")), nr, nth, prec,
                           max(1, min(_log(rng, 4, 200), int(cap))), consistent=opt, exponents=opt), name="drawn solve")
    if kind == "sector":
        nr = _log(rng, 2000, 24000)
        return _solve("drawn sector", rng.choice(("sector", "planar")), nr, 1, prec, _log(rng, 100, 400))
    if kind == "host":
        nr, nth = _log(rng, 256, 1200), _log(rng, 256, 1200)
        return _solve("drawn host", rng.choice(("explosion", "implosion")), nr, nth, "fp32", _log(rng, 4, 40),
                      kind="host")
    if kind == "batch":
        prec = rng.choice(("fp32", "fp32", "fp32", "fp64"))
        return {"name": "drawn batch", "kind": "batch", "instances": rng.randint(4, 28), "nmin": _log(rng, 64, 128),
                "nmax": _log(rng, 160, 640 if prec == "fp32" else 200), "precision": prec,
                "steps": _log(rng, 32, 96 if prec == "fp32" else 48)}
    if kind == "serve":
        return {"name": "drawn serve", "kind": "serve", "instances": rng.randint(2, 9), "nmin": 128,
                "nmax": _log(rng, 160, 512), "precision": "fp32", "steps": _log(rng, 100, 400)}
    return {"name": "drawn " + kind, "kind": kind, "nr": _log(rng, 64, 2000), "ntheta": _log(rng, 64, 2000),
            "precision": prec}


# ---------------------------------------------------------------------------
# parameters and seeded fields
# ---------------------------------------------------------------------------
def _params(case):
    nr, nth, shape = case["nr"], case["ntheta"], case.get("shape", "explosion")
    kw = dict(nr=nr, ntheta=nth, precision=case["precision"])
    if shape == "sector":
        kw.update(r_in=0.0, r_out=5e-5 * nr, dt=1.25e-6, tau=2e-4, omega1=1.0, omega2=50.0, sector=1,
                  r_bc_inner="centre")
        return W.base_params(**kw)
    if shape == "planar":
        kw.update(r_in=1000.0, r_out=1000.0 + 5e-6 * nr, dt=2.5e-7, tau=2e-4, omega1=10.0, omega2=1000.0, sector=1)
        return W.base_params(**kw)
    r_in = 0.05
    dr, dth = 1.0 / nr, 2.0 * math.pi / nth
    # Courant sum at most 0.57 at the innermost radius, and the benchmark's dt at its size
    kw.update(r_in=r_in, r_out=r_in + 1.0, dt=min(1e-5, 0.4 * min(dr, r_in * dth) / 12.5), tau=1e-3,
              omega1=0.0 if shape == "inert" else 2.0, omega2=0.0 if shape == "inert" else 2.0)
    if case.get("consistent"):
        kw.update(reaction_energy=1)
    if case.get("exponents"):
        kw.update(m=1.5, n=0.7)
    return W.base_params(**kw)


def _grid(p):
    dev = _device()
    dr = (p["r_out"] - p["r_in"]) / p["nr"]
    span = math.pi / 4.0 if p.get("sector") else 2.0 * math.pi
    r = p["r_in"] + (torch.arange(p["nr"], dtype=torch.float64, device=dev) + 0.5) * dr
    th = torch.arange(p["ntheta"], dtype=torch.float64, device=dev) * (span / p["ntheta"])
    return r, th, dr, span / p["ntheta"]


def _fields(p, shape, seed):
    """[5][ntheta][nr] FP64 fields: a hot ring or a shocked, perturbed outer ring
    beside fresh gas, with 1 % density noise."""
    dev = _device()
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    r, th, _, _ = _grid(p)
    x = ((r - p["r_in"]) / (p["r_out"] - p["r_in"]))[None, :]
    if shape == "implosion":
        phase = 2.0 * math.pi * torch.rand(13, dtype=torch.float64, device=dev, generator=gen)
        q = torch.arange(4, 17, dtype=torch.float64, device=dev)
        front = 0.85 * (1.0 + 0.005 * torch.cos(q[None, :] * th[:, None] + phase[None, :]).mean(1))[:, None]
        hot, driver = x > front, (1.4, -0.5, 0.0, 1.6, 1.0)
    elif shape == "inert":
        hot, driver = (x < 0.25) & (th[:, None] < 10.0), (2.0, 0.0, 0.0, 2.0, 0.0)
    elif shape == "sector":
        hot, driver = (x < 0.1) & (th[:, None] < 10.0), (1.5, 0.666667, 0.0, 1.55556, 1.0)
    elif shape == "planar":
        hot, driver = (x < 0.1) & (th[:, None] < 10.0), (1.35826, 0.81650, 0.0, 2.59709, 1.0)
    else:
        hot, driver = (x < 0.2) & (th[:, None] < 10.0), (1.4, 0.0, 0.0, 1.6, 1.0)
    fresh = (1.0, 0.0, 0.0, 1.0, 0.0)
    out = torch.empty((5, p["ntheta"], p["nr"]), dtype=torch.float64, device=dev)
    for k in range(5):
        out[k].fill_(fresh[k])
        out[k][hot] = driver[k]
    noise = torch.rand((p["ntheta"], p["nr"]), dtype=torch.float64, device=dev, generator=gen)
    out[0] *= 1.0 + 0.01 * (2.0 * noise - 1.0)
    return out


def _raw_state(case, seed):
    """A state away from equilibrium (f^eq of the fields, each f off by up to
    5 %) in the case's precision: parameters, f, stored lambda."""
    p = _params(case)
    fields = _fields(p, "implosion", seed)
    gen = torch.Generator(device=_device())
    gen.manual_seed(int(seed) + 1)
    f, lam = _init64(p, fields)
    for q in range(NV):
        f[q] *= 1.0 + 0.05 * (2.0 * torch.rand(f[q].shape, dtype=torch.float64, device=f.device, generator=gen) - 1.0)
    dt = torch.float64 if case["precision"] == "fp64" else torch.float32
    return p, f.to(dt), (lam if case["precision"] == "fp64" else 1.0 - lam).to(dt)


def _instances(case, seed):
    """(parameters, fields, steps) of each simulation of a sweep or of a request stream."""
    n = case["instances"]
    u = W.uniform(7, 20, 2 * n)  # the sizes are the case's, the fields the seed's
    got = []
    for i in range(n):
        N = case["nmin"] + int(u[i] * (case["nmax"] - case["nmin"] + 1))
        steps = case["steps"]
        if case["kind"] == "serve":
            N = max(32, N // 32 * 32)
            steps = max(1, int(steps * (0.5 + 0.5 * u[n + i])))
        shape = "explosion" if i % 2 == 0 else "implosion"
        one = _solve("", shape, N, N, case["precision"], steps)
        p = _params(one)
        got.append((p, _fields(p, shape, int(seed) * 64 + i), steps))
    return got


# ---------------------------------------------------------------------------
# prepare and run
# ---------------------------------------------------------------------------
def _state_views(sim):
    """f [33][ntheta][nr] of the simulation's current state, in place."""
    f_at, _, ld = sim.state_device()
    nth, nr = sim.shape
    real = torch.float64 if sim.p.precision == dbm.DBM_FP64 else torch.float32
    first = f_at - sim.buf.data_ptr()
    size = NV * nth * ld * (8 if real == torch.float64 else 4)
    return sim.buf[first:first + size].view(real).view(NV, nth, ld)[:, :, :nr]


def prepare(case, seed):
    kind, dev = case["kind"], _device()
    if kind in ("solve", "host"):
        p = _params(case)
        fields = _fields(p, case["shape"], seed)
        st = {"case": case, "sim": dbm.Simulation(p)}
        if kind == "solve":
            st["fields"] = fields
            st["out"] = torch.empty((5, p["ntheta"], p["nr"]), dtype=torch.float64, device=dev)
        else:
            st["host"] = [torch.empty(fields[k].shape, dtype=torch.float64, pin_memory=True).copy_(fields[k])
                          for k in range(5)]
            st["host_out"] = [torch.empty(fields[k].shape, dtype=torch.float64, pin_memory=True) for k in range(5)]
        return st
    if kind == "batch":
        got = _instances(case, seed)
        return {"case": case, "sims": [dbm.Simulation(p) for p, _, _ in got], "fields": [f for _, f, _ in got],
                "out": [torch.empty((5, p["ntheta"], p["nr"]), dtype=torch.float64, device=dev) for p, _, _ in got],
                "batch": dbm.Batch(case["instances"], 1 << 15, case["precision"])}
    if kind == "serve":
        got = _instances(case, seed)
        requests = [(dbm.params_from(p), dict(zip(FIELDS, f.cpu().numpy())), steps) for p, f, steps in got]
        return {"case": case, "requests": requests,
                "server": dbm.Server(768 << 20, max_slots=8, quantum=64, precision=case["precision"])}
    p, f, lam = _raw_state(case, seed)
    sim = dbm.Simulation(p)
    sim.import_state(f.cpu().numpy(), lam.cpu().numpy(), 0)
    shape = (p["ntheta"], p["nr"])
    return {"case": case, "sim": sim, "out": torch.empty((5,) + shape, dtype=torch.float64, device=dev),
            "noneq": torch.empty((12,) + shape, dtype=torch.float64, device=dev)}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        sim, out = state["sim"], state["out"]
        dbm.dbm_init_state_device(sim.h, state["fields"].data_ptr())
        sim.step(case["steps"])
        dbm.dbm_moments_device(sim.h, out.data_ptr())
        return {"moments": out, "f": _state_views(sim)}
    if kind == "host":
        sim = state["sim"]
        dbm.dbm_init_state(sim.h, *[a.numpy() for a in state["host"]])
        sim.step(case["steps"])
        totals = np.zeros(4)
        dbm.dbm_moments(sim.h, *[a.numpy() for a in state["host_out"]], totals=totals)
        return {"moments": state["host_out"], "totals": totals}
    if kind == "batch":
        batch, sims = state["batch"], state["sims"]
        for slot, (sim, fields) in enumerate(zip(sims, state["fields"])):
            dbm.dbm_init_state_device(sim.h, fields.data_ptr())
            batch.attach(slot, sim, case["steps"])
        batch.step(case["steps"])
        for slot, (sim, out) in enumerate(zip(sims, state["out"])):
            batch.detach(slot)
            dbm.dbm_moments_device(sim.h, out.data_ptr())
        return state["out"]
    if kind == "serve":
        server = state["server"]
        tickets = [server.submit(p, fields, steps) for p, fields, steps in state["requests"]]
        done = [server.poll(t) for t in tickets]
        return [{k: r[k] for k in FIELDS} for _, r in done]
    sim = state["sim"]
    dbm.dbm_noneq_device(sim.h, state["noneq"].data_ptr())
    if kind == "noneq":
        return {"noneq": state["noneq"]}
    dbm.dbm_moments_device(sim.h, state["out"].data_ptr())
    return {"moments": state["out"], "noneq": state["noneq"]}


def work(case):
    """Bytes: the fields or the state read once, the fields (and state) written
    once.  Flops of one site's step: 13 per velocity (equilibrium 8, collision
    and streaming 5 multiply-adds and products, counted 19 flops) and some 200
    for moments, coefficients and lambda."""
    per_step = 19 * 32 + 200
    kind, wide = case["kind"], 8 if case.get("precision") == "fp64" else 4
    if kind in ("solve", "host"):
        sites = case["nr"] * case["ntheta"]
        return {"bytes": sites * (40 + 40 + (NV * wide if kind == "solve" else 0)),
                "flops": float(sites) * case["steps"] * per_step}
    if kind in ("batch", "serve"):
        sites = work_sites(case)
        return {"bytes": sum(s for s, _ in sites) * 80, "flops": float(sum(s * n for s, n in sites)) * per_step}
    sites = case["nr"] * case["ntheta"]
    out = 96 if kind == "noneq" else 136
    return {"bytes": sites * ((NV + (kind == "diagnose")) * wide + out), "flops": float(sites) * (NV * 8 + 150)}


def work_sites(case):
    n, u = case["instances"], W.uniform(7, 20, 2 * case["instances"])
    got = []
    for i in range(n):
        N, steps = case["nmin"] + int(u[i] * (case["nmax"] - case["nmin"] + 1)), case["steps"]
        if case["kind"] == "serve":
            N, steps = max(32, N // 32 * 32), max(1, int(steps * (0.5 + 0.5 * u[n + i])))
        got.append((N * N, steps))
    return got


# ---------------------------------------------------------------------------
# the update in plain torch, 64 bits
# ---------------------------------------------------------------------------
def _velocities(p):
    v = torch.tensor([0.0] + [s for s in p["v"] for _ in range(8)], dtype=torch.float64, device=_device())
    i = torch.tensor([0] + list(range(8)) * 4, dtype=torch.float64, device=_device())
    return v, i * (math.pi / 4.0)


def _polar(p):
    """v_r, v_theta: [33][ntheta]."""
    v, ang = _velocities(p)
    _, th, _, _ = _grid(p)
    return v[:, None] * torch.cos(ang[:, None] - th[None, :]), v[:, None] * torch.sin(ang[:, None] - th[None, :])


def _weights(p, T):
    x = [s * s for s in p["v"]]
    F = []
    for k in range(4):
        a, b, c = (x[(k + s) % 4] for s in (1, 2, 3))
        F.append((48.0 * T ** 4 - 6.0 * (a + b + c) * T ** 3 + (a * b + b * c + c * a) * T ** 2
                  - 0.25 * a * b * c * T) / (x[k] * (x[k] - a) * (x[k] - b) * (x[k] - c)))
    return [1.0 - 8.0 * sum(F)] + F


def _moments(vr, vth, f):
    rho = f.sum(0)
    ur = torch.einsum("qm,qmj->mj", vr, f) / rho
    uth = torch.einsum("qm,qmj->mj", vth, f) / rho
    T = torch.zeros_like(rho)
    for q in range(NV):
        T += 0.5 * f[q] * ((vr[q][:, None] - ur) ** 2 + (vth[q][:, None] - uth) ** 2)
    return rho, ur, uth, T / rho


def _feq(F, vr, vth, q, rho, ur, uth, T):
    u2 = ur * ur + uth * uth
    xi = (vr[q][:, None] * ur + vth[q][:, None] * uth) / T
    h = 1.0 - u2 / (2.0 * T)
    return rho * F[0 if q == 0 else 1 + (q - 1) // 8] * (
        h + u2 * u2 / (8.0 * T * T) + xi * h + 0.5 * xi * xi * h + xi ** 3 / 6.0 + xi ** 4 / 24.0)


def _init64(p, fields):
    vr, vth = _polar(p)
    rho, ur, uth, T, lam = fields
    F = _weights(p, T)
    return torch.stack([_feq(F, vr, vth, q, rho, ur, uth, T) for q in range(NV)]), lam.clone()


def _turn(q, s):
    return 0 if q == 0 else 1 + (q - 1) // 8 * 8 + ((q - 1) % 8 + s) % 8


def _step64(p, f, lam, vr, vth):
    r, _, dr, dth = _grid(p)
    dt, sector, centre = p["dt"], p.get("sector", 0), p.get("r_bc_inner") == "centre"
    rho, ur, uth, T = _moments(vr, vth, f)
    F = _weights(p, T)
    P, burns = rho * T, T > p["T_th"]
    zero = torch.zeros_like(P)
    a = torch.where(burns, p["omega1"] * P ** p["m"], zero)
    b = torch.where(burns, p["omega2"] * P ** p["n"], zero)
    R = (1.0 - lam) * (a + b * lam)
    grow = torch.expm1((a + b) * dt)
    low = (a + b) + (a + b * lam) * grow
    dlam = torch.where(low > 0.0, R * grow / torch.where(low > 0.0, low, zero + 1.0), zero)
    if p.get("reaction_energy"):
        R = dlam / dt
    decay = math.exp(-dt / p["tau"])
    new = torch.empty_like(f)
    for q in range(NV):
        g = f[q]
        feq = _feq(F, vr, vth, q, rho, ur, uth, T)
        c2 = (vr[q][:, None] - ur) ** 2 + (vth[q][:, None] - uth) ** 2
        t = feq + (g - feq) * decay + dt * feq * (c2 - 2.0 * T) / (2.0 * T * T) * p["Q"] * R
        cr = vr[q][:, None] * (dt / dr)
        ct = vth[q][:, None] * dt / (r[None, :] * dth)
        inner = f[_turn(q, 4)][:, :1] if centre else g[:, :1]
        back = torch.cat([inner, g[:, :-1]], 1)
        fore = torch.cat([g[:, 1:], g[:, -1:]], 1)
        below = torch.cat([f[_turn(q, 1) if sector else q][-1:], g[:-1]], 0)
        above = torch.cat([g[1:], f[_turn(q, -1) if sector else q][:1]], 0)
        t -= torch.where(cr >= 0.0, cr * (g - back), cr * (fore - g))
        t -= torch.where(ct >= 0.0, ct * (g - below), ct * (above - g))
        new[q] = t
    lb, lf = torch.cat([lam[:, :1], lam[:, :-1]], 1), torch.cat([lam[:, 1:], lam[:, -1:]], 1)
    ld, lu = torch.roll(lam, 1, 0), torch.roll(lam, -1, 0)
    ln = lam + dlam - ur * (dt / dr) * torch.where(ur >= 0.0, lam - lb, lf - lam)
    ln -= uth * dt / (r[None, :] * dth) * torch.where(uth >= 0.0, lam - ld, lu - lam)
    return new, ln.clamp(0.0, 1.0)


def _solve64(p, fields, steps):
    vr, vth = _polar(p)
    f, lam = _init64(p, fields)
    for _ in range(steps):
        f, lam = _step64(p, f, lam, vr, vth)
    return torch.stack(list(_moments(vr, vth, f)) + [lam]), f


def _noneq64(p, f):
    vr, vth = _polar(p)
    rho, ur, uth, T = _moments(vr, vth, f)
    M = torch.zeros((12,) + rho.shape, dtype=torch.float64, device=f.device)
    for q in range(NV):
        a, b, g = vr[q][:, None] - ur, vth[q][:, None] - uth, f[q]
        h = 0.5 * (a * a + b * b)
        for c, w in enumerate((a * a, a * b, b * b, a * a * a, a * a * b, a * b * b, b * b * b, h * a, h * b,
                               h * a * a, h * a * b, h * b * b)):
            M[c] += g * w
    for c in (0, 2):
        M[c] -= rho * T
    for c in (9, 11):
        M[c] -= 2.0 * rho * T * T
    return M


def exact(case, seed):
    kind = case["kind"]
    if kind in ("solve", "host"):
        p = _params(case)
        if p["nr"] * p["ntheta"] * case["steps"] + 2e5 * case["steps"] > 2e8:
            return None
        moments, f = _solve64(p, _fields(p, case["shape"], seed), case["steps"])
        return {"moments": moments, "f": f} if kind == "solve" else {"moments": list(moments), "totals": None}
    if kind in ("batch", "serve"):
        sites = work_sites(case)
        if sum((s + 2e5) * n for s, n in sites) > 9e8:
            return None
        got = [_solve64(p, fields, steps)[0] for p, fields, steps in _instances(case, seed)]
        return got if kind == "batch" else [dict(zip(FIELDS, m)) for m in got]
    p, f, lam = _raw_state(case, seed)
    f, lam = f.double(), lam.double()
    noneq = _noneq64(p, f)
    if kind == "noneq":
        return {"noneq": noneq}
    vr, vth = _polar(p)
    lam = lam if case["precision"] == "fp64" else 1.0 - lam
    return {"moments": torch.stack(list(_moments(vr, vth, f)) + [lam]), "noneq": noneq}
