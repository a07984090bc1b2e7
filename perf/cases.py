"""Performance cases of the lattice step, through the package's public entry points.

Each case is a piece of work that a user's program has the library do: a few steps of a lattice or of
a batch and the fields read back (`carry`: the state goes on from pass to pass, as in a program that
alternates steps and snapshots), or a whole solve segment, initial fields in, steps, fields out.  Host
arrays are pinned, as the benchmark's are.  Fields of an FP32 lattice come back from the library
widened to 64 bits; the cases keep them in 32 bits, the precision they have.

`exact` advances the same inputs in 64 bits with plain torch operations on whole fields (the method's
equations as the paper states them: arXiv 2009.05264, Sec. 2), independently of the library.
"""
import math
import random

import numpy as np
import torch

from paper_2009_05264_gb300 import lbm

DEVICE = "cuda" if torch.cuda.is_available() else "cpu"
DEFAULTS = dict(thermal=1, members=0, carry=0, hazi=0, bubbles=0, two_phase=0, records=0)


# ---------------------------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------------------------
def listed():
    cases = [
        # watching a static droplet (the isothermal FP64 droplet of the validation runs): a few steps
        # at a time on a lattice so small that launches and latency are all there is
        dict(name="droplet 128x128 fp64", geometry="periodic", nx=128, ny=128, precision="fp64", thermal=0, steps=5,
             carry=1, two_phase=1),
        # a thermal two-phase drop in a periodic box, FP32: wraps on every side, an odd width
        dict(name="thermal drop 251x190 fp32", geometry="periodic", nx=251, ny=190, precision="fp32", steps=60,
             two_phase=1),
        # contact-angle calibration: a batch of sessile drops, isothermal, walls, snapshots of the density
        dict(name="sessile batch 6x 100x50 fp32", geometry="walls", nx=100, ny=50, members=6, precision="fp32",
             thermal=0, steps=200, carry=1, two_phase=1),
        # pool boiling at six gravities, advanced as one batch between density snapshots
        dict(name="pool batch 6x 128x512 fp32", geometry="pool", nx=128, ny=512, members=6, precision="fp32",
             steps=100, carry=1),
        # the boiling channel of the departure statistics: vapour counters on, every step's record read
        dict(name="boiling 600x80 fp32", geometry="channel", nx=600, ny=80, precision="fp32", steps=250, bubbles=1,
             records=1),
        # the paper-sized channel, in both precisions
        dict(name="channel 1000x100 fp32", geometry="channel", nx=1000, ny=100, precision="fp32", steps=500),
        dict(name="channel 1000x100 fp64", geometry="channel", nx=1000, ny=100, precision="fp64", steps=100),
        # the other energy source (Hazi-Markus), ragged in both directions
        dict(name="hazi channel 777x67 fp32", geometry="channel", nx=777, ny=67, precision="fp32", steps=200, hazi=1),
        # a served request of the larger kind
        dict(name="channel 4000x400 fp32", geometry="channel", nx=4000, ny=400, precision="fp32", steps=200),
        # a parameter sweep: 64 channels of uneven size in one batch
        dict(name="sweep batch 64 fp32", geometry="channel", nx=2000, ny=200, members=64, precision="fp32", steps=150,
             carry=1),
        # FP64 at a size that fills the GPU
        dict(name="channel 4000x800 fp64", geometry="channel", nx=4000, ny=800, precision="fp64", steps=30),
        # the benchmark channel
        dict(name="channel 8000x800 fp32", geometry="channel", nx=8000, ny=800, precision="fp32", steps=200),
    ]
    return [dict(DEFAULTS, **c) for c in cases]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["droplet", "drop", "sessile", "pool", "boiling", "channel", "channel", "channel", "walls", "hazi",
                       "sweep"])
    prec = rng.choice(["fp32", "fp32", "fp32", "fp64"])
    if kind == "droplet":
        n = log_int(48, 300)
        return dict(DEFAULTS, geometry="periodic", nx=n, ny=log_int(48, 300), precision=rng.choice(["fp64", "fp32"]),
                    thermal=0, steps=log_int(1, 30), carry=1, two_phase=1)
    if kind == "drop":
        return dict(DEFAULTS, geometry="periodic", nx=log_int(64, 700), ny=log_int(64, 500), precision=prec,
                    steps=log_int(10, 60), two_phase=1)
    if kind == "sessile":
        return dict(DEFAULTS, geometry="walls", nx=log_int(80, 260), ny=log_int(40, 130), members=rng.randint(2, 12),
                    precision="fp32", thermal=0, steps=log_int(50, 200), carry=1, two_phase=1)
    if kind == "pool":
        nx = log_int(64, 200)
        return dict(DEFAULTS, geometry="pool", nx=nx, ny=4 * nx, members=rng.randint(1, 8), precision="fp32",
                    steps=log_int(25, 150), carry=1)
    if kind == "boiling":
        return dict(DEFAULTS, geometry="channel", nx=log_int(300, 1200), ny=log_int(50, 120), precision=prec,
                    steps=log_int(50, 250), bubbles=1, records=1)
    if kind == "walls":
        return dict(DEFAULTS, geometry="walls", nx=log_int(100, 3000), ny=log_int(30, 300), precision=prec,
                    steps=log_int(20, 100))
    if kind == "hazi":
        return dict(DEFAULTS, geometry="channel", nx=log_int(200, 3000), ny=log_int(40, 200), precision=prec,
                    steps=log_int(20, 200), hazi=1)
    if kind == "sweep":
        nx = log_int(500, 2000)
        return dict(DEFAULTS, geometry="channel", nx=nx, ny=log_int(60, 200), members=rng.randint(3, 48),
                    precision="fp32", steps=log_int(16, 100), carry=1)
    nx, ny = log_int(150, 8000), log_int(20, 800)
    most = (3.2e8 if prec == "fp32" else 4e7) / (nx * ny)  # steps that keep below the largest cases
    return dict(DEFAULTS, geometry="channel", nx=nx, ny=ny, precision=prec, steps=max(4, min(500, log_int(4, 500), int(most))))


def members_of(case):
    """(nx, ny, parameter overrides) of every lattice of a case, from the case alone."""
    if not case["members"]:
        return [(case["nx"], case["ny"], {})]
    rng = random.Random(case["nx"] * 1009 + case["ny"])
    out = []
    for k in range(case["members"]):
        if case["geometry"] == "walls":  # contact angles: one wall density per drop
            out.append((case["nx"], case["ny"], dict(rho_w=2.2 + 1.8 * k / max(1, case["members"] - 1))))
        elif case["geometry"] == "pool":  # one gravity per pool
            out.append((case["nx"], case["ny"], dict(g_a=1e-4 * 10 ** (k / max(1, case["members"] - 1)))))
        else:  # a sweep over size, inlet velocity, superheat and wettability
            out.append((rng.randint(max(3, case["nx"] // 5), case["nx"]), rng.randint(max(2, case["ny"] // 4), case["ny"]),
                        dict(u_in=rng.uniform(0.01, 0.028), dTheat_R=rng.uniform(0.03, 0.1), rho_w=rng.uniform(2.6, 4.0))))
    return out


RHO_L, RHO_V = 5.88, 0.59  # coexisting densities at 0.9 Tc as the paper prints them
PR = dict(a=2.0 / 49.0, b=2.0 / 21.0, R=1.0, omega=0.32, beta=1.16, c0=6.0, G=-1.0, tau_f=1.0, tau_g=0.6, c_v=6.0)
TC = 0.0778 * PR["a"] / (0.45724 * PR["b"] * PR["R"])


def parameters(case, nx, extra):
    """Every parameter that a case's lattice runs with (the library's names)."""
    p = dict(PR, geometry=case["geometry"], thermal=case["thermal"], multiphase=1, T0_R=0.9, Tin_R=0.9, u_in=0.03,
             dTheat_R=0.08, heater_x0=nx // 5, heater_len=max(5, min(40, nx // 4)), heat_on_step=0, g_a=5e-5,
             rho_out=5.95, rho_w=5.95, init_rho_out=5.95, source_model=case["hazi"], bubble_stats=case["bubbles"],
             rho_vapor=3.2)
    if case["geometry"] == "pool":
        p.update(rho_out=RHO_L, init_rho_out=RHO_L, rho_w=3.0, u_in=0.0, dTheat_R=0.3, heater_x0=nx // 2 - 5,
                 heater_len=10)
    if case["bubbles"]:
        p.update(rho_out=RHO_L, init_rho_out=RHO_L, rho_w=3.0, u_in=0.005, dTheat_R=0.3, g_a=2e-4)
    if case["two_phase"]:
        p.update(init_rho_out=RHO_L, rho_out=RHO_L, g_a=0.0 if not case["thermal"] else 5e-5, heater_len=0)
    p.update(extra)
    p["G_wet"] = 9.0 * (1.0 + p["beta"]) * p["G"]
    return p


def initial_fields(case, nx, ny, seed):
    """(rho, ux, uy, T) in 64 bits: a liquid with smooth seeded waves and noise, or a drop in vapour."""
    g = torch.Generator(device=DEVICE).manual_seed(int(seed) * 7919 + nx * 31 + ny)
    ph = torch.rand(8, generator=g, device=DEVICE, dtype=torch.float64) * (2 * math.pi)
    noise = torch.rand((ny, nx), generator=g, device=DEVICE, dtype=torch.float64) * 2 - 1
    y = torch.arange(ny, device=DEVICE, dtype=torch.float64)[:, None]
    x = torch.arange(nx, device=DEVICE, dtype=torch.float64)[None, :]
    sx, sy = 2 * math.pi / nx, 2 * math.pi / ny
    # a drop is carried along at the inlet velocities of the sweeps, unless it rests on a wall
    du = 0.05 if case["two_phase"] and case["geometry"] == "periodic" else 0.005
    ux = du * torch.sin(sy * y + ph[2]) * torch.cos(sx * x + ph[3])
    uy = du * torch.sin(sx * x + ph[4]) * torch.sin(sy * y + ph[5])
    T = 0.9 * TC * (1 + 0.002 * torch.cos(sx * x + ph[6]) * torch.sin(sy * y + ph[7]))
    if case["two_phase"]:
        wall = case["geometry"] == "walls"
        cx, cy, r0 = (nx - 1) / 2, -0.5 if wall else (ny - 1) / 2, 0.36 * ny if wall else 0.2 * min(nx, ny)
        r = torch.sqrt((x - cx) ** 2 + (y - cy) ** 2)
        rho = (RHO_L + RHO_V) / 2 - (RHO_L - RHO_V) / 2 * torch.tanh(2.0 * (r - r0) / 2.0)
        rho = rho * (1 + 1e-3 * noise)
    else:
        rho0 = RHO_L if case["bubbles"] or case["geometry"] == "pool" else 5.95
        rho = rho0 * (1 + 0.002 * (torch.sin(sx * x + ph[0]) * torch.cos(sy * y + ph[1]) + 0.1 * noise))
    return tuple(v.expand(ny, nx) for v in (rho, ux, uy, T))


# ---------------------------------------------------------------------------------------------
# what is timed
# ---------------------------------------------------------------------------------------------
def wanted(case):
    """The fields that the program reads: calibration and pools follow the density (and the temperature)."""
    if not case["members"]:
        return ("rho", "ux", "uy", "T") if case["thermal"] else ("rho", "ux", "uy")
    return {"walls": ("rho",), "pool": ("rho", "T"), "channel": ("rho", "ux", "uy", "T")}[case["geometry"]]


def pinned(n):
    t = torch.empty(n, dtype=torch.float64)
    return t.pin_memory() if torch.cuda.is_available() else t


def prepare(case, seed):
    todo = members_of(case)
    nodes = sum(nx * ny for nx, ny, _ in todo)
    st = dict(case=case, out={k: pinned(nodes) for k in wanted(case)}, lats=[], fields=[], views=[], batch=None)
    if case["members"]:
        st["batch"] = lbm.Batch(case["precision"], thermal=bool(case["thermal"]))
    at = 0
    for m, (nx, ny, extra) in enumerate(todo):
        p = parameters(case, nx, extra)
        if st["batch"] is not None:
            lat = st["batch"].add(nx, ny, p)
        else:
            lat = lbm.Lattice(nx, ny, case["precision"])
            lat.set_params(p)
        host = []
        for v in initial_fields(case, nx, ny, int(seed) * 64 + m):
            h = pinned(nx * ny)
            h.copy_(v.reshape(-1))
            host.append(h.numpy().reshape(ny, nx))
        if case["carry"]:
            lat.init_fields(*host)
        else:
            st["fields"].append(host)
        st["lats"].append(lat)
        st["views"].append({k: t[at : at + nx * ny].numpy().reshape(ny, nx) for k, t in st["out"].items()})
        at += nx * ny
    return st


def run(st):
    case, lats = st["case"], st["lats"]
    if not case["carry"]:
        for lat, host in zip(lats, st["fields"]):
            lat.init_fields(*host)
    first = lats[0].step_count
    (st["batch"] or lats[0]).step(case["steps"])
    records = lats[0].diagnostics_range(first, case["steps"]) if case["records"] else None
    for lat, views in zip(lats, st["views"]):
        lat.fields(out=views)
    kind = torch.float32 if case["precision"] == "fp32" else torch.float64
    out = {k: t.to(kind) for k, t in st["out"].items()}
    if "ux" in out:  # the velocity, one vector field
        out["u"] = torch.stack((out.pop("ux"), out.pop("uy")))
    if records is not None:
        out["records"] = torch.from_numpy(records).to(kind)
    return out


def work(case):
    """A step's state (9 or 18 populations a node) read once and written once per step, initial fields in and
    fields out once a pass; the arithmetic of one node update, counted as additions and multiplications."""
    nodes = sum(nx * ny for nx, ny, _ in members_of(case))
    elt = 8 if case["precision"] == "fp64" else 4
    pops = 18 if case["thermal"] else 9
    io = 8 * nodes * ((0 if case["carry"] else 4) + len(wanted(case)))
    return {"bytes": nodes * case["steps"] * 2 * pops * elt + io,
            "flops": nodes * case["steps"] * (400 if case["thermal"] else 250)}


# ---------------------------------------------------------------------------------------------
# the same in 64 bits with plain torch
# ---------------------------------------------------------------------------------------------
CX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
CY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
WT = (4 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 9, 1 / 36, 1 / 36, 1 / 36, 1 / 36)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)


def _equilibrium(m, ux, uy):
    uu = ux * ux + uy * uy
    out = []
    for i in range(9):
        cu = CX[i] * ux + CY[i] * uy
        out.append(WT[i] * m * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu))
    return torch.stack(out)


class _Plain:
    def __init__(self, p, fields):
        self.p, self.geo = p, p["geometry"]
        rho, ux, uy, T = fields
        self.ny, self.nx = rho.shape
        self.f, self.g = _equilibrium(rho, ux, uy), _equilibrium(T, ux, uy)
        self.mean, self.rho_prev, self.n = rho.mean(), rho.clone(), 0
        w = p["omega"]
        self.kappa = 0.37464 + 1.54226 * w - 0.26992 * w * w
        self.T0, self.Tin, self.Thot = 0.9 * TC, 0.9 * TC, (0.9 + p["dTheat_R"]) * TC
        self.psi_w = self.psi(torch.tensor(float(p["rho_w"]), dtype=torch.float64), torch.tensor(self.T0, dtype=torch.float64)).item()

    def pressure(self, rho, T):
        p = self.p
        s = 1 + self.kappa * (1 - torch.sqrt(T / TC))
        return rho * p["R"] * T / (1 - p["b"] * rho) - p["a"] * s * s * rho * rho / (
            1 + 2 * p["b"] * rho - (p["b"] * rho) ** 2)

    def psi(self, rho, T):
        return torch.sqrt(2 * (self.pressure(rho, T) - rho / 3) / (self.p["c0"] * self.p["G"]))

    def ghosts(self, v, solid=0.0):
        """v with one ghost node on each side: wraps, the end column at open ends, `solid` behind a wall."""
        if self.geo == "channel":
            v = torch.cat((v[:, :1], v, v[:, -1:]), 1)
        else:
            v = torch.cat((v[:, -1:], v, v[:, :1]), 1)
        if self.geo == "periodic":
            return torch.cat((v[-1:], v, v[:1]), 0)
        row = torch.full_like(v[:1], solid)
        return torch.cat((row, v, v[-1:] if self.geo == "pool" else row), 0)

    def macroscopic(self):
        p, f = self.p, self.f
        rho = f.sum(0)
        ux = (f[1] - f[3] + f[5] - f[6] - f[7] + f[8]) / rho
        uy = (f[2] - f[4] + f[5] + f[6] - f[7] - f[8]) / rho
        T = self.g.sum(0) if p["thermal"] else torch.full_like(rho, self.T0)
        psi = self.psi(rho, T)
        pad = self.ghosts(psi)
        Fx, Fy = torch.zeros_like(rho), torch.zeros_like(rho)
        for i in range(1, 9):
            G = (2.0 if i <= 4 else 0.5) * p["G"]
            q = pad[1 + CY[i] : 1 + CY[i] + self.ny, 1 + CX[i] : 1 + CX[i] + self.nx]
            term = -p["beta"] * psi * G * q - 0.5 * (1 - p["beta"]) * G * q * q
            Fx = Fx + CX[i] * term
            Fy = Fy + CY[i] * term
        if self.geo != "periodic":  # sum of w_i c_i over the wall's sites is (0, -1/6), or (0, 1/6) at the top
            Fy[0] += p["G_wet"] * psi[0] * self.psi_w / 6
            if self.geo != "pool":
                Fy[-1] -= p["G_wet"] * psi[-1] * self.psi_w / 6
        Fy = Fy - (rho - self.mean) * p["g_a"]
        return rho, ux, uy, T, Fx, Fy, ux + Fx / (2 * rho), uy + Fy / (2 * rho)

    def hot(self, step, sx):
        """Bottom-wall temperature at the sites sx."""
        on = self.p["thermal"] and self.p["heater_len"] > 0 and step >= self.p["heat_on_step"]
        lo = self.p["heater_x0"]
        hot = ((sx >= lo) & (sx < lo + self.p["heater_len"]) & bool(on)).double()
        return self.Tin + hot * (self.Thot - self.Tin)

    def step(self):
        p, f, g, nx, ny = self.p, self.f, self.g, self.nx, self.ny
        rho, ux, uy, T, Fx, Fy, ax, ay = self.macroscopic()
        eq = _equilibrium(rho, ux, uy)
        fs = f - (f - eq) / p["tau_f"] + _equilibrium(rho, ux + Fx / rho, uy + Fy / rho) - eq
        gs = g
        if p["thermal"]:
            padx, pady = self.ghosts(ax), self.ghosts(ay)
            dyu = 0.5 * (pady[2:, 1:-1] - pady[:-2, 1:-1])
            if self.geo != "periodic":
                dyu[0] = ay[1] - ay[0]
                if self.geo != "pool":
                    dyu[-1] = ay[-1] - ay[-2]
            div = 0.5 * (padx[1:-1, 2:] - padx[1:-1, :-2]) + dyu
            s = 1 + self.kappa * (1 - torch.sqrt(T / TC))
            dalpha = -self.kappa * s / torch.sqrt(T * TC)
            dpdT = rho * p["R"] / (1 - p["b"] * rho) - p["a"] * dalpha * rho * rho / (1 + 2 * p["b"] * rho - (p["b"] * rho) ** 2)
            if p["source_model"]:
                phi = T / (rho * rho * p["c_v"]) * dpdT * (rho - self.rho_prev) + T * div
            else:
                phi = T * (1 - dpdT / (rho * p["c_v"])) * div
            w = torch.tensor(WT, dtype=torch.float64, device=f.device)[:, None, None]
            gs = g - (g - _equilibrium(T, ax, ay)) / p["tau_g"] + w * phi
        record = self.record(rho, T, ax)
        self.mean, self.rho_prev = rho.mean(), rho
        fn = torch.stack([torch.roll(fs[i], (CY[i], CX[i]), (0, 1)) for i in range(9)])
        gn = torch.stack([torch.roll(gs[i], (CY[i], CX[i]), (0, 1)) for i in range(9)]) if p["thermal"] else g
        if self.geo != "periodic":
            x = torch.arange(nx, device=f.device)
            for i in (2, 5, 6):
                sx = x - CX[i] if self.geo == "channel" else (x - CX[i]) % nx
                fn[i][0] = fs[OPP[i]][0]
                if p["thermal"]:
                    gn[i][0] = -gs[OPP[i]][0] + 2 * WT[i] * self.hot(self.n, sx)
            for i in (4, 7, 8) if self.geo != "pool" else ():
                fn[i][-1] = fs[OPP[i]][-1]
                if p["thermal"]:
                    gn[i][-1] = -gs[OPP[i]][-1] + 2 * WT[i] * self.Tin
        if self.geo == "channel":
            self.open_ends(fn, gn, gs)
        if self.geo == "pool":
            self.surface(fn, gn)
        self.f, self.g, self.n = fn, gn, self.n + 1
        return record

    def open_ends(self, f, g, gs):
        p = self.p
        c, u = f[:, :, 0], p["u_in"]  # inlet: u = (u_in, 0)
        ru = u * (c[0] + c[2] + c[4] + 2 * (c[3] + c[6] + c[7])) / (1 - u)
        f1 = c[3] + 2 / 3 * ru
        f5 = c[7] - 0.5 * (c[2] - c[4]) + ru / 6
        f8 = c[6] + 0.5 * (c[2] - c[4]) + ru / 6
        keep5, keep8 = c[5, 0].clone(), c[8, -1].clone()  # corners: the link from the wall is known
        f5[0], f8[-1] = keep5, keep8
        for row, known in ((0, 5), (-1, 8)):
            k = c[:, row]
            a, b = (f5[row], k[2] + k[6] + f5[row] - k[4] - k[7]) if known == 5 else (k[4] + k[7] + f8[row] - k[2] - k[6], f8[row])
            # sum of f is rho, of f c_x is rho u: rho from both, f1 from the second
            rest = k[0] + k[2] + k[3] + k[4] + k[6] + k[7] + a + b
            mom = a + b - k[3] - k[6] - k[7]
            r = (rest - mom) / (1 - u)
            f5[row], f8[row], f1[row] = a, b, r * u - mom
        f[1, :, 0], f[5, :, 0], f[8, :, 0] = f1, f5, f8
        c, r = f[:, :, -1], p["rho_out"]  # outlet: rho = rho_out, u_y = 0
        ru = c[0] + c[2] + c[4] + 2 * (c[1] + c[5] + c[8]) - r
        f3 = c[1] - 2 / 3 * ru
        f7 = c[5] + 0.5 * (c[2] - c[4]) - ru / 6
        f6 = c[8] - 0.5 * (c[2] - c[4]) - ru / 6
        f6[0], f7[0] = c[6, 0], c[2, 0] + c[5, 0] + c[6, 0] - c[4, 0] - c[8, 0]
        f7[-1], f6[-1] = c[7, -1], c[4, -1] + c[7, -1] + c[8, -1] - c[2, -1] - c[5, -1]
        for row in (0, -1):
            f3[row] = r - (c[0, row] + c[1, row] + c[2, row] + c[4, row] + c[5, row] + c[8, row] + f6[row] + f7[row])
        f[3, :, -1], f[6, :, -1], f[7, :, -1] = f3, f6, f7
        if p["thermal"]:
            top, low = slice(0, -1), slice(1, None)  # rows where the link does not come from a wall
            g[1, :, 0] = -gs[3, :, 0] + 2 * WT[1] * self.Tin
            g[5, low, 0] = -gs[7, low, 0] + 2 * WT[5] * self.Tin
            g[8, top, 0] = -gs[6, top, 0] + 2 * WT[8] * self.Tin
            g[:, :, -1] = g[:, :, -2]

    def surface(self, f, g):
        c, r = f[:, -1], self.p["rho_out"]
        ru = c[0] + c[1] + c[3] + 2 * (c[2] + c[5] + c[6]) - r
        h = 0.5 * (c[1] - c[3])
        f4, f7, f8 = c[2] - 2 / 3 * ru, c[5] + h - ru / 6, c[6] - h - ru / 6
        f[4, -1], f[7, -1], f[8, -1] = f4, f7, f8
        g[:, -1] = g[:, -2]

    def record(self, rho, T, ax):
        p, nx, ny = self.p, self.nx, self.ny
        z = torch.zeros((), dtype=torch.float64, device=rho.device)
        dp = dt = fin = fout = z
        if self.geo == "channel":
            pr = [self.pressure(rho[ny // 2, x], T[ny // 2, x]) for x in (1, nx - 2)]
            dp, fin, fout = pr[0] - pr[1], (rho[:, 0] * ax[:, 0]).sum(), (rho[:, -1] * ax[:, -1]).sum()
        lo, hi = p["heater_x0"], p["heater_x0"] + p["heater_len"]
        if self.geo != "periodic" and p["thermal"] and p["heater_len"] and self.n >= p["heat_on_step"]:
            dt = (self.Thot - T[0, lo:hi].mean()) / (self.Thot - T.mean())
        vap = (rho < p["rho_vapor"]).double() * p["bubble_stats"]
        wall = vap[0].sum() if self.geo != "periodic" else z
        heat = vap[0, lo:hi].sum() if self.geo != "periodic" else z
        zone = vap[:, max(0, lo - p["heater_len"]) : lo + 2 * p["heater_len"]].sum()
        return torch.stack([z + self.n, rho.sum(), T.sum(), rho.mean(), dp, dt, fin, fout, vap.sum(), wall, heat, zone])


def exact(case, seed):
    out, records = {k: [] for k in wanted(case)}, []
    for m, (nx, ny, extra) in enumerate(members_of(case)):
        sim = _Plain(parameters(case, nx, extra), initial_fields(case, nx, ny, int(seed) * 64 + m))
        for _ in range(case["steps"]):
            rec = sim.step()
            if case["records"]:
                records.append(rec)
        rho, _, _, T, _, _, ax, ay = sim.macroscopic()
        for k, v in (("rho", rho), ("ux", ax), ("uy", ay), ("T", T)):
            if k in out:
                out[k].append(v.reshape(-1).cpu())
    out = {k: torch.cat(v) for k, v in out.items()}
    if "ux" in out:
        out["u"] = torch.stack((out.pop("ux"), out.pop("uy")))
    if case["records"]:
        out["records"] = torch.stack(records).cpu()
    return out
