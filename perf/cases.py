"""The work that the boiling framework is timed on: single domains stepped from a
given state, batches of domains, gradients of the wall heat flux, and field
read-outs, each through the calls of paper_1501_03857_gb300.lb.

A stepping pass puts the given state (populations and temperature, on the
device) into the simulation, advances it, and reads the state and the heat-flux
statistics back, as a program does that evaluates windows from saved states; so
every pass does the same work on the same data.
"""

import math
from functools import lru_cache

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1501_03857_gb300 import inputs, lb

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
M_ROWS = ((1, 1, 1, 1, 1, 1, 1, 1, 1), (-4, -1, -1, -1, -1, 2, 2, 2, 2), (4, -2, -2, -2, -2, 1, 1, 1, 1),
          (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, -2, 0, 2, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1),
          (0, 0, -2, 0, 2, 1, 1, -1, -1), (0, 1, -1, 1, -1, 0, 0, 0, 0), (0, 0, 0, 0, 0, 1, -1, 1, -1))
BC = {"walls": lb.BC_WALLS, "outflow": lb.BC_TOP_OUTFLOW, "periodic": lb.BC_PERIODIC}
# wettabilities of the sessile-droplet range (about 45 to 150 degrees)
GW_VALUES = (0.0, 0.03, 0.065, 0.09, 0.105)


def _case(name, kind, Lx, Ly, steps, layout="pool", bc="walls", ghost=False, isothermal=False, superheat=0.0137,
          Gw=0.0, **more):
    return dict({"name": name, "kind": kind, "Lx": Lx, "Ly": Ly, "steps": steps, "layout": layout, "bc": bc,
                 "ghost": ghost, "isothermal": isothermal, "superheat": superheat, "Gw": Gw}, **more)


def listed():
    return [
        # one control interval on the paper's own pool (Sec. 3.1): a new wall
        # temperature profile, one step, the flux back; latency decides
        _case("control_600x150", "control", 600, 150, 1, superheat=0.0165, Gw=0.065),
        # the smallest pool in use (quick checks, parameter scans): launches decide
        _case("pool_100x100", "step", 100, 100, 64, bc="outflow", superheat=0.0109),
        # the paper's pool between two samples of a single run
        _case("pool_600x150", "step", 600, 150, 128, Gw=0.065),
        # a tall odd-sized domain with the open top and the ghost-layer wall
        _case("outflow_517x1003", "step", 517, 1003, 64, bc="outflow", ghost=True, superheat=0.0109, Gw=0.03),
        # the large bubble-array domain of the benchmark
        _case("bubbles_4096x4096", "step", 4096, 4096, 32, layout="bubbles", superheat=0.0109),
        # the contact-angle calibration: isothermal sessile droplets, one per G_w
        _case("droplets_11x240x120", "batch", 240, 120, 64, layout="droplet", isothermal=True, superheat=0.0,
              n=11, uneven=False, persistent=0, block=128),
        # the benchmark's boiling curve: 48 domains of uneven sizes, one launch a step
        _case("curve_48_uneven", "batch", 400, 600, 32, superheat=0.044, n=48, uneven=True, persistent=0, block=128),
        # the paper's curves: 36 cases of the 600 x 150 pool in the persistent launch
        _case("curve_36x600x150", "batch", 600, 150, 64, superheat=0.023, n=36, uneven=False, persistent=1, block=64),
        # gradient of the window's mean flux, every step stored (the default choice)
        _case("adjoint_256x256", "adjoint", 256, 256, 128, superheat=0.0109, Gw=0.05, ckpt=1),
        # the same on the paper's pool from checkpoints, when memory is short
        _case("adjoint_600x150_ckpt", "adjoint", 600, 150, 96, superheat=0.0137, Gw=0.065, ckpt=8),
        # the gradient on a large domain
        _case("adjoint_2048x2048", "adjoint", 2048, 2048, 8, layout="bubbles", superheat=0.0109, Gw=0.05, ckpt=1),
        # macroscopic fields and the mass of a large domain, as sampled during a run
        _case("fields_2048x2048", "fields", 2048, 2048, 0, layout="bubbles", superheat=0.0109, Gw=0.065),
    ]


def draw(rng):
    kind = rng.choice(["step", "step", "step", "batch", "adjoint", "fields", "control"])

    def logsize(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    bc = rng.choice(["walls", "walls", "outflow", "periodic"]) if kind in ("step", "fields") else \
        rng.choice(["walls", "walls", "outflow"])
    ghost = bc != "periodic" and rng.random() < 0.3
    superheat, Gw = round(rng.uniform(0.008, 0.02), 4), rng.choice(GW_VALUES)
    cells = math.exp(rng.uniform(math.log(100 * 100), math.log({"step": 4000 ** 2, "control": 2000 ** 2, "batch": 400 ** 2,
                                                               "adjoint": 1800 ** 2, "fields": 2900 ** 2}[kind])))
    aspect = math.exp(rng.uniform(math.log(0.4), math.log(4.0)))
    Lx, Ly = max(int(round(math.sqrt(cells * aspect))), 60), max(int(round(math.sqrt(cells / aspect))), 48)
    layout = "bubbles" if min(Lx, Ly) >= 400 and rng.random() < 0.6 else "pool"
    more = {}
    if kind == "step":
        steps = min(128, max(16, int(4.5e8 / (Lx * Ly))))
        more = {"isothermal": rng.random() < 0.2}
    elif kind == "control":
        steps = 1
        bc = "walls"
    elif kind == "batch":
        n = logsize(4, 48)
        steps = min(96, max(32, int(1.6e8 / (n * Lx * Ly))))
        bc, layout, mode = "walls", "pool", rng.choice([(0, 128), (0, 64), (1, 64), (2, 128)])
        uneven = Lx >= 200 and Ly >= 200 and rng.random() < 0.5
        if uneven:
            Lx, Ly = 400, 600  # the ranges of the uneven sizes
            steps = 32
        more = {"isothermal": (not uneven) and rng.random() < 0.3, "n": n, "uneven": uneven, "persistent": mode[0],
                "block": mode[1]}
    elif kind == "adjoint":
        steps = min(96, max(6, int(2.5e7 / (Lx * Ly))))
        more = {"ckpt": rng.choice([1, 1, 4, 8])}
    else:
        steps = 0
    c = _case("", kind, Lx, Ly, steps, layout=layout, bc=bc, ghost=ghost, superheat=superheat, Gw=Gw, **more)
    del c["name"]
    return c


# ---- inputs --------------------------------------------------------------------


def _pr(eos):
    Tc = 0.0778 * eos["a"] / (0.45724 * eos["b"] * eos["R"])
    om = eos["omega"]
    return Tc, 0.37464 + 1.54226 * om - 0.26992 * om * om


EOS = {"a": 3 / 49, "b": 2 / 21, "R": 1.0, "omega": 0.344}


@lru_cache(maxsize=None)
def coexistence(Ts_over_Tc=0.86):
    """Maxwell equal-area densities (rho_V, rho_L) of the Peng-Robinson EOS."""
    a, b, R = EOS["a"], EOS["b"], EOS["R"]
    Tc, kap = _pr(EOS)
    T = Ts_over_Tc * Tc
    ph = (1 + kap * (1 - math.sqrt(T / Tc))) ** 2

    def p(r):
        return r * R * T / (1 - b * r) - a * ph * r * r / (1 + 2 * b * r - b * b * r * r)

    def prim(v):
        s = math.sqrt(2.0)
        return R * T * math.log(v - b) - a * ph / (2 * s * b) * math.log((v + b - s * b) / (v + b + s * b))

    g = np.linspace(1e-6, 0.999 / b, 40001)
    d = np.diff(p(g))
    k = np.nonzero(np.sign(d[:-1]) != np.sign(d[1:]))[0]
    r_hi, r_lo = g[k[0] + 1], g[k[1] + 1]

    def root(P, lo, hi):
        up = p(hi) > P
        for _ in range(200):
            m = 0.5 * (lo + hi)
            if (p(m) > P) == up:
                hi = m
            else:
                lo = m
        return 0.5 * (lo + hi)

    P0, P1 = max(p(r_lo), 1e-8 * p(r_hi)), p(r_hi)
    for _ in range(200):
        P = 0.5 * (P0 + P1)
        vv, vl = 1 / root(P, 1e-18, r_hi), 1 / root(P, r_lo, (1 / b) * (1 - 1e-9))
        if prim(vv) - prim(vl) - P * (vv - vl) > 0:
            P0 = P
        else:
            P1 = P
    return 1 / vv, 1 / vl


def _density(layout, Lx, Ly, periodic, g, dev):
    """Smooth-interface density [Ly, Lx] (float64): a rippled pool (60 % of
    the height, as the paper's 90 of 150), vapour bubbles in liquid (radii 20
    to 60, smaller in small domains), or a sessile droplet."""
    rv, rl = coexistence()
    x = torch.arange(Lx, device=dev, dtype=torch.float64)[None, :]
    y = torch.arange(Ly, device=dev, dtype=torch.float64)[:, None]
    u = torch.rand(16, generator=g, device=dev, dtype=torch.float64).tolist()
    mid, amp = 0.5 * (rl + rv), 0.5 * (rl - rv)
    if layout == "pool" and periodic:  # a liquid slab between two interfaces
        rho = rv + amp * (torch.tanh(2.0 * (y - 0.2 * Ly) / 5.0) - torch.tanh(2.0 * (y - 0.75 * Ly) / 5.0)) + 0.0 * x
    elif layout == "pool":
        h = 0.6 * Ly + min(4.0, 0.03 * Ly) * sum(torch.sin(2 * math.pi * (k * x / Lx + u[k])) / k for k in (1, 2, 3))
        rho = mid - amp * torch.tanh(2.0 * (y - h) / 5.0)
    elif layout == "droplet":
        R = min(40.0, 0.3 * Ly) * (0.9 + 0.2 * u[0])
        dx = (x - Lx * (0.4 + 0.2 * u[1])).abs()
        dx = torch.minimum(dx, Lx - dx)
        rho = mid - amp * torch.tanh(2.0 * (torch.sqrt(dx * dx + y * y) - R) / 5.0)
    else:
        rho = torch.full((Ly, Lx), rl, device=dev, dtype=torch.float64)
        rmax = min(60.0, min(Lx, Ly) / 8.0)
        n = max(1, int(256 * Lx * Ly / 4096.0 ** 2))
        c = torch.rand(n, 3, generator=g, device=dev, dtype=torch.float64).tolist()
        for cu, cv, cr in c:
            r = rmax * (1 / 3 + 2 / 3 * cr)
            cx, cy = cu * Lx, r + 24 + cv * max(Ly - 2 * (r + 24), 0.0)
            x0, x1 = int(cx - r - 20), int(cx + r + 21)
            y0, y1 = max(int(cy - r - 20), 0), min(int(cy + r + 21), Ly)
            xs = torch.arange(x0, x1, device=dev)
            d = torch.sqrt((xs - cx)[None, :] ** 2 + (y[y0:y1] - cy) ** 2)
            dip = rl - amp * (1.0 - torch.tanh(2.0 * (d - r) / 5.0))
            cols = xs % Lx
            rho[y0:y1, cols] = torch.minimum(rho[y0:y1, cols], dip)
    return rho * (1.0 + 1e-3 * (2 * torch.rand(Ly, Lx, generator=g, device=dev, dtype=torch.float64) - 1))


def _domain(c, seed, Lx, Ly, superheat, Gw):
    """One domain's inputs, float32 on the device: rho0, populations near
    equilibrium in a smooth flow (speeds up to about 0.02), theta = T - T_s
    (a heated layer on the wall), the wall profile and the scalars."""
    dev = "cuda"
    g = torch.Generator(device=dev)
    g.manual_seed(seed)
    per = c["bc"] == "periodic"
    rho = _density(c["layout"], Lx, Ly, per, g, dev).float()
    u = torch.rand(16, generator=g, device=dev, dtype=torch.float64).tolist()
    x = torch.arange(Lx, device=dev, dtype=torch.float32)[None, :] * (2 * math.pi / Lx)
    y = torch.arange(Ly, device=dev, dtype=torch.float32)[:, None]
    env = torch.cos(y * (2 * math.pi / Ly)) if per else torch.sin(y * (math.pi / (Ly - 1)))
    ux = 0.008 * env * (torch.sin(x + 6.28 * u[0]) + torch.sin(3 * x + 6.28 * u[1]))
    uy = 0.008 * env * (torch.cos(2 * x + 6.28 * u[2]) + torch.cos(5 * x + 6.28 * u[3]))
    f = torch.empty(9, Ly, Lx, device=dev)
    for a in range(9):
        eu = EX[a] * ux + EY[a] * uy
        f[a] = WT[a] * rho * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * (ux * ux + uy * uy))
        f[a] *= 1 + 1e-3 * (2 * torch.rand(Ly, Lx, generator=g, device=dev) - 1)
    prof = 0.2 * superheat * np.sin(2 * np.pi * (np.arange(Lx) / Lx + u[4]))
    th = torch.zeros(Ly, Lx, device=dev)
    if not c["isothermal"]:
        th += superheat * (1 + 0.2 * torch.sin(2 * x + 6.28 * u[5])) * (0.3 * (1 + torch.cos(y * (2 * math.pi / Ly)))
                                                                    if per else torch.exp(-y / 8.0))
        th *= 1 + 0.02 * (2 * torch.rand(Ly, Lx, generator=g, device=dev) - 1)
    if not per:
        th[0] = torch.from_numpy((superheat + prof).astype(np.float32)).to(dev)
        th[-1] = 0.0
    return {"rho0": rho.cpu().numpy(), "f": f, "th": th, "prof": prof, "superheat": superheat, "Gw": Gw, "Lx": Lx,
            "Ly": Ly}


def _config(c, Lx, Ly):
    return lb.Config(Lx=Lx, Ly=Ly, bc_y=BC[c["bc"]], ghost_layer=c["ghost"], isothermal=c["isothermal"],
                     g=0.0 if c["layout"] == "droplet" else 3e-5)


def _domains(c, seed):
    if c["kind"] != "batch":
        return [_domain(c, seed, c["Lx"], c["Ly"], c["superheat"], c["Gw"])]
    if c["uneven"]:  # the benchmark's sizes
        sizes = [(d["Lx"], d["Ly"]) for d in inputs.boiling_curve_batch(n=c["n"], lx_range=(200, c["Lx"]),
                                                                       ly_range=(200, c["Ly"]))]
    else:
        sizes = [(c["Lx"], c["Ly"])] * c["n"]
    return [_domain(c, seed * 1000 + i, Lx, Ly, c["superheat"] * (0.4 + 0.6 * i / max(c["n"] - 1, 1)),
                    GW_VALUES[i % len(GW_VALUES)]) for i, (Lx, Ly) in enumerate(sizes)]


def prepare(case, seed):
    doms = _domains(case, seed)
    s = {"case": case, "doms": doms}
    n = sum(d["f"][0].numel() for d in doms)
    if case["kind"] == "batch":
        s["batch"] = lb.Batch([{"cfg": _config(case, d["Lx"], d["Ly"]), "superheat": d["superheat"], "Gw": d["Gw"],
                                "profile": d["prof"], "rho0": d["rho0"]} for d in doms])
        s["batch"].set_launch(case["block"], 0)
        if case["persistent"]:
            s["batch"].set_persistent(case["persistent"])
    else:
        d = doms[0]
        s["sim"] = lb.Simulation(_config(case, d["Lx"], d["Ly"]), superheat=d["superheat"], Gw=d["Gw"],
                                 profile=d["prof"], rho0=d["rho0"])
    for d in doms:
        del d["rho0"]
    if case["kind"] == "fields":
        lb.check(lb.lib.lb_set_state(s["sim"].h, doms[0]["f"].data_ptr(), doms[0]["th"].data_ptr(), 1))
        s["out"] = [torch.empty(doms[0]["Ly"], doms[0]["Lx"], device="cuda") for _ in range(4)]
    else:
        s["fout"] = torch.empty(9 * n, device="cuda")
        s["tout"] = torch.empty(n, device="cuda")
    return s


# ---- the passes -----------------------------------------------------------------


def run(s):
    return _RUN[s["case"]["kind"]](s)


def _set(sim, d):
    lb.check(lb.lib.lb_set_state(sim.h, d["f"].data_ptr(), d["th"].data_ptr(), 1))


def _state(s):
    d = s["doms"][0]
    f, th = s["fout"].view(9, d["Ly"], d["Lx"]), s["tout"].view(d["Ly"], d["Lx"])
    s["sim"].get_state_device(f, th)
    return {"f": f, "theta": th}


def _run_step(s):
    sim = s["sim"]
    _set(sim, s["doms"][0])
    sim.step(s["case"]["steps"])
    q = sim.heat_flux(reset=True)
    return dict(_state(s), q_inst=q["q_inst"], q_mean=q["q_mean"])


def _run_control(s):
    sim, d = s["sim"], s["doms"][0]
    _set(sim, d)
    sim.set_wall_temperature(1.1 * d["superheat"], d["prof"])
    sim.step(1)
    return dict(_state(s), q_inst=sim.heat_flux(reset=True)["q_inst"])


def _run_batch(s):
    b = s["batch"]
    for i, d in enumerate(s["doms"]):
        lb.check(lb.lib.lb_batch_set_state(b.h, i, d["f"].data_ptr(), d["th"].data_ptr(), 1))
    b.step(s["case"]["steps"])
    at = 0
    for i, d in enumerate(s["doms"]):
        lb.check(lb.lib.lb_batch_get_state(b.h, i, s["fout"].data_ptr() + 36 * at, s["tout"].data_ptr() + 4 * at, 1))
        at += d["Lx"] * d["Ly"]
    q = b.heat_flux(reset=True)
    return {"f": s["fout"], "theta": s["tout"], "q_mean": q["q_mean"].tolist()}


def _run_adjoint(s):
    sim = s["sim"]
    _set(sim, s["doms"][0])
    J, dTb, dGw = sim.adjoint(s["case"]["steps"], s["case"]["ckpt"])
    # the gradient as an optimiser of a float32 wall profile takes it (heat_flux_window's form)
    return dict(_state(s), J=J, dTb=torch.as_tensor(dTb, dtype=torch.float32, device="cuda"), dGw=dGw)


def _run_fields(s):
    s["sim"].fields_device(*s["out"])
    return {"rho": s["out"][0], "ux": s["out"][1], "uy": s["out"][2], "T": s["out"][3], "mass": s["sim"].mass()}


_RUN = {"step": _run_step, "control": _run_control, "batch": _run_batch, "adjoint": _run_adjoint,
        "fields": _run_fields}


def work(case):
    """Bytes: a step reads and writes nine populations and a temperature in
    FP32; a reverse step reads the state and the adjoint state and writes the
    adjoint state; fields read the state and write four planes, the mass reads
    the populations. A pass puts the state in and reads it back (each a copy).
    Flops: about 400 a cell and step, 900 a cell and reverse step."""
    if case["kind"] == "batch" and case["uneven"]:
        cells = sum(d["Lx"] * d["Ly"] for d in inputs.boiling_curve_batch(
            n=case["n"], lx_range=(200, case["Lx"]), ly_range=(200, case["Ly"])))
    else:
        cells = case["Lx"] * case["Ly"] * case.get("n", 1)
    n = case["steps"]
    if case["kind"] == "fields":
        return {"bytes": cells * (40 + 16 + 36), "flops": cells * 100}
    if case["kind"] == "adjoint":
        return {"bytes": cells * (200 * n + 160), "flops": cells * 1300 * n}
    return {"bytes": cells * (80 * n + 160), "flops": cells * 400 * n}


# ---- the same in 64 bits, in plain torch -------------------------------------------


class _Model:
    """The method's constants and one time step in float64; fields are
    [..., Ly, Lx], populations [9, ..., Ly, Lx]."""

    def __init__(self, c, d, rho_ave, Gw):
        self.c, self.per = c, c["bc"] == "periodic"
        self.Tc, self.kap = _pr(EOS)
        self.Ts = 0.86 * self.Tc
        self.rv, self.rl = coexistence()
        self.rho_ave, self.Gw = rho_ave, Gw
        self.g = 0.0 if c["layout"] == "droplet" else 3e-5
        y = torch.arange(d["Ly"], device="cuda")[:, None]
        no = torch.zeros_like(y, dtype=torch.bool)
        self.bot, self.top = (no, no) if self.per else (y == 0, y == d["Ly"] - 1)
        self.first = no if self.per else y == 1
        self.wall = self.bot | self.top
        M = torch.tensor(M_ROWS, dtype=torch.float64, device="cuda")
        self.M, self.Mi = M, torch.linalg.inv(M)

    def psi(self, rho, T):
        a, b, R = EOS["a"], EOS["b"], EOS["R"]
        ph = (1 + self.kap * (1 - torch.sqrt(T / self.Tc))) ** 2
        p = rho * R * T / (1 - b * rho) - a * ph * rho * rho / (1 + 2 * b * rho - b * b * rho * rho)
        return torch.sqrt(-2.0 * (p - rho / 3))

    def near(self, v, ghost=False):
        """v(x + e_a) for a = 0..8."""
        if ghost and not self.per:
            v = torch.cat([v[..., :1, :], v, v[..., -1:, :]], -2)
            return [torch.roll(v, (-EY[a], -EX[a]), (-2, -1))[..., 1:-1, :] for a in range(9)]
        return [torch.roll(v, (-EY[a], -EX[a]), (-2, -1)) for a in range(9)]

    @staticmethod
    def grad(nb):
        d1, d2 = nb[5] - nb[7], nb[8] - nb[6]
        return (nb[1] - nb[3]) / 3 + (d1 + d2) / 12, (nb[2] - nb[4]) / 3 + (d1 - d2) / 12

    @staticmethod
    def lap(nb):
        return (2 / 3) * (nb[1] + nb[2] + nb[3] + nb[4]) + (1 / 6) * (nb[5] + nb[6] + nb[7] + nb[8]) - (10 / 3) * nb[0]

    def flow(self, fs, th):
        bot, top = self.bot, self.top
        f = [torch.roll(fs[a], (EY[a], EX[a]), (-2, -1)) for a in range(9)]
        if not self.per:
            d = 0.5 * (f[1] - f[3])
            f[2] = torch.where(bot, f[4], f[2])
            f[5] = torch.where(bot, f[7] - d, f[5])
            f[6] = torch.where(bot, f[8] + d, f[6])
            if self.c["bc"] == "walls":
                f[4] = torch.where(top, f[2], f[4])
                f[7] = torch.where(top, f[5] + d, f[7])
                f[8] = torch.where(top, f[6] - d, f[8])
            else:
                for a in (4, 7, 8):
                    f[a] = torch.where(top, torch.roll(fs[a], EX[a], -1), f[a])
        f = torch.stack(f)
        rho = f.sum(0)
        psi = self.psi(rho, self.Ts + th)
        gx, gy = self.grad(self.near(psi, True))
        Fmx, Fmy = psi * gx, psi * gy  # G = -1
        if not self.c["ghost"]:
            Fmx, Fmy = Fmx.masked_fill(self.wall, 0.0), Fmy.masked_fill(self.wall, 0.0)
        body = -(rho - self.rho_ave) * self.g + torch.where(self.first, self.Gw / 6 * psi * psi, torch.zeros_like(psi))
        Fx, Fy = Fmx, Fmy + body.masked_fill(self.wall, 0.0)
        jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7])
        jy = (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8])
        return f, rho, psi, Fmx, Fmy, Fx, Fy, (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho

    def step(self, fs, th, tb):
        """(f*, theta) of the next level and q(t)."""
        f, rho, psi, Fmx, Fmy, Fx, Fy, vx, vy = self.flow(fs, th)
        m = torch.tensordot(self.M, f, 1)
        v2 = vx * vx + vy * vy
        meq = torch.stack([rho, rho * (-2 + 3 * v2), rho * (1 - 3 * v2), rho * vx, -rho * vx, rho * vy, -rho * vy,
                           rho * (vx * vx - vy * vy), rho * vx * vy])
        s_e, s_z, s_q, sigma = 0.8, 0.8, 1.1, 1.2
        ratio, vF = (Fmx * Fmx + Fmy * Fmy) / (psi * psi), vx * Fx + vy * Fy
        S = torch.stack([torch.zeros_like(rho), 6 * vF + sigma * ratio / (1 / s_e - 0.5),
                         -6 * vF - sigma * ratio / (1 / s_z - 0.5), Fx, -Fx, Fy, -Fy, 2 * (vx * Fx - vy * Fy),
                         vx * Fy + vy * Fx])
        tl, tv = 0.8, 1.0  # 3 nu + 1/2 for nu_L = 0.1, nu_V = 0.5/3
        snu = 1 / (tv + (tl - tv) * torch.clamp((rho - self.rv) / (self.rl - self.rv), 0, 1))
        one = torch.ones_like(rho)
        lam = torch.stack([one, s_e * one, s_z * one, one, s_q * one, one, s_q * one, snu, snu])
        fn = torch.tensordot(self.Mi, m - lam * (m - meq) + (1 - 0.5 * lam) * S, 1)
        q = (-0.028 * rho[..., 0, :] * (-3 * th[..., 0, :] + 4 * th[..., 1, :] - th[..., 2, :]) / 2).mean(-1)
        if self.c["isothermal"]:
            return fn, th, q
        a, b, R, cv, chi = EOS["a"], EOS["b"], EOS["R"], 6.0, 0.028 / 6.0
        drx, dry = self.grad(self.near(rho))
        div = self.grad(self.near(vx))[0] + self.grad(self.near(vy))[1]
        fluid = (~self.wall).double()

        def rhs(t):
            nb = self.near(t)
            gx, gy = self.grad(nb)
            T = self.Ts + t
            dphi = -self.kap * (1 + self.kap * (1 - torch.sqrt(T / self.Tc))) / torch.sqrt(T * self.Tc)
            dpdT = rho * R / (1 - b * rho) - a * dphi * rho * rho / (1 + 2 * b * rho - b * b * rho * rho)
            return fluid * (-(vx * gx + vy * gy) + chi * (self.lap(nb) + (drx * gx + dry * gy) / rho)
                            - T / (rho * cv) * dpdT * div)

        h1 = rhs(th)
        h2 = rhs(th + 0.5 * h1)
        h3 = rhs(th + 0.5 * h2)
        h4 = rhs(th + h3)
        tn = th + (h1 + 2 * h2 + 2 * h3 + h4) / 6
        if not self.per:
            tn = torch.where(self.bot, tb[..., None, :], tn).masked_fill(self.top, 0.0)
        return fn, tn, q


def exact(case, seed):
    doms = _domains(case, seed)
    if case["kind"] == "batch" and not case["uneven"]:  # equal sizes: all at once
        d = dict(doms[0], f=torch.stack([x["f"] for x in doms], 1), th=torch.stack([x["th"] for x in doms]))
        col = lambda v: torch.tensor(v, dtype=torch.float64, device="cuda")[:, None, None]  # noqa: E731
        d["rho_ave"] = col([float(x["rho0"].mean(dtype=np.float64)) for x in doms])
        d["Gw"] = col([x["Gw"] for x in doms])
        d["tb"] = torch.from_numpy(np.stack([x["superheat"] + x["prof"] for x in doms])).cuda()
        f, th, qs = _steps(case, d)
        n = len(doms)
        return {"f": f.transpose(0, 1).reshape(-1), "theta": th.reshape(-1), "q_mean": qs.mean(0).reshape(n).tolist()}
    out = []
    for d in doms:
        d["rho_ave"] = float(d["rho0"].mean(dtype=np.float64))
        k = 1.1 if case["kind"] == "control" else 1.0
        d["tb"] = torch.from_numpy(k * d["superheat"] + d["prof"]).cuda()
        out.append(_EXACT[case["kind"]](case, d))
    if case["kind"] == "batch":
        return {"f": torch.cat([o["f"].reshape(-1) for o in out]), "theta": torch.cat([o["theta"].reshape(-1) for o in out]),
                "q_mean": [o["q_mean"] for o in out]}
    return out[0]


def _steps(case, d):
    m = _Model(case, d, d["rho_ave"], d["Gw"])
    f, th, qs = d["f"].double(), d["th"].double(), []
    if case["kind"] == "control":  # the new profile replaces the wall row at once
        th[0] = d["tb"]
    for _ in range(case["steps"]):
        f, th, q = m.step(f, th, d["tb"])
        qs.append(q)
    return f, th, torch.stack(qs)


def _exact_step(case, d):
    f, th, qs = _steps(case, d)
    none = case["bc"] == "periodic"  # no wall, no flux
    return {"f": f, "theta": th, "q_inst": 0.0 if none else float(qs[-1]), "q_mean": 0.0 if none else float(qs.mean())}


def _exact_control(case, d):
    f, th, qs = _steps(case, d)
    return {"f": f, "theta": th, "q_inst": float(qs[-1])}


def _exact_adjoint(case, d):
    tb = d["tb"].clone().requires_grad_()
    gw = torch.tensor(d["Gw"], dtype=torch.float64, device="cuda", requires_grad=True)
    m = _Model(case, d, d["rho_ave"], gw)
    f, th = d["f"].double(), torch.cat([tb[None], d["th"].double()[1:]])
    qs = []
    for _ in range(case["steps"]):
        f, th, q = checkpoint(m.step, f, th, tb, use_reentrant=False)
        qs.append(q)
    J = torch.stack(qs).mean()
    gtb, ggw = torch.autograd.grad(J, (tb, gw))
    return {"f": f.detach(), "theta": th.detach(), "J": float(J.detach()), "dTb": gtb, "dGw": float(ggw)}


def _exact_fields(case, d):
    m = _Model(case, d, d["rho_ave"], d["Gw"])
    f, th = d["f"].double(), d["th"].double()
    _, rho, _, _, _, _, _, vx, vy = m.flow(f, th)
    return {"rho": rho, "ux": vx, "uy": vy, "T": m.Ts + th, "mass": float(f.sum())}


_EXACT = {"step": _exact_step, "control": _exact_control, "batch": _exact_step, "adjoint": _exact_adjoint,
          "fields": _exact_fields}
