"""Performance cases of the boiling-flow library: the runs its users make, through its public Python API.

A case is a plain dict; prepare() builds the simulation a program would keep, run() makes one pass
of that program's loop (steps, then the heat flux and the fields it looks at), and exact() gives the
same outputs from a plain FP64 torch restatement of the method, written here from its equations.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1912_02018_gb300 import Batch, Sim

U_IN = 0.05


# ---------------------------------------------------------------- the cases
def _cyl(name, nx, ny, D, Re, dT, steps, build="f32", boil=True, xf=0.25, a_num=2, psi_mode=0):
    return {"name": name, "kind": "step", "nx": nx, "ny": ny, "D": float(D), "xf": xf, "Re": float(Re), "dT": dT,
            "steps": steps, "build": build, "boil": boil, "a_num": a_num, "psi_mode": psi_mode}


def _shear(name, L, Ma, Re, collision, steps, build="f32"):
    return {"name": name, "kind": "shear", "L": L, "Ma": Ma, "Re": Re, "collision": collision, "steps": steps,
            "build": build}


def _batch(name, Ds, W, H, a_num, steps, build="f32"):
    return {"name": name, "kind": "batch", "Ds": Ds, "W": W, "H": H, "a_num": a_num, "steps": steps, "build": build}


def _adjoint(name, nx, ny, D, Re, dT, steps, ckpt, build="f32", boil=True):
    return {"name": name, "kind": "adjoint", "nx": nx, "ny": ny, "D": float(D), "xf": 0.25, "Re": float(Re), "dT": dT,
            "steps": steps, "ckpt": ckpt, "build": build, "boil": boil, "a_num": 2, "psi_mode": 0}


def listed():
    return [
        # the smallest domain people run (parity, parameter studies, long runs of 50,000 steps): launches and latency
        _cyl("small_128x64", 128, 64, 16, 30, 0.05, 20, boil=False),
        # the paper's own domain (20 D x 45 D, D = 30, flow along x): neither side a multiple of a tile
        _cyl("paper_1350x600", 1350, 600, 30, 30, 0.05, 20, xf=0.2, a_num=3),
        # one domain of the Reynolds-superheat sweep
        _cyl("sweep_1536x768", 1536, 768, 96, 300, 0.10, 20),
        # the benchmark's workload: film boiling at high Reynolds number
        _cyl("film_2048x1024", 2048, 1024, 128, 30000, 0.20, 20, boil=False),
        # a production-sized lattice, far larger than the L2
        _cyl("large_8192x4096", 8192, 4096, 512, 30000, 0.20, 4, boil=False),
        # populations stored as shifted FP16 (half the state and half the checkpoint)
        _cyl("f16s_1536x768", 1536, 768, 96, 3000, 0.10, 20, build="f16s"),
        # the FP64 build, which reference runs are made with
        _cyl("f64_512x256", 512, 256, 32, 300, 0.05, 10, build="f64"),
        # double shear layer: periodic, single phase, the collision pass alone
        _shear("shear_512", 512, 0.1, 3.0e4, 0, 50),
        # boiling-curve sweep over domains of uneven size, stepped together
        _batch("batch16_uneven", "64,40,128,96,40,64,64,128,96,40,40,96,64,128,40,64", 12, 6, 2, 20),
        # the paper's boiling curve: thirteen superheats on its domain, stepped together
        _batch("batch13_paper", ",".join(["30"] * 13), 45, 20, 3, 10),
        # gradient of the window-mean heat flux for design and inverse problems, FP32 and FP64
        _adjoint("adjoint_512x256", 512, 256, 32, 300, 0.05, 250, 50),
        _adjoint("adjoint_f64_256x128", 256, 128, 32, 300, 0.05, 100, 25, build="f64"),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(("step", "shear", "batch", "adjoint"), (62, 10, 14, 14))[0]
    if kind == "shear":
        L = int(_log(rng, 64, 2048))
        build = rng.choices(("f32", "f64"), (4, 1))[0]
        if build == "f64":
            L = min(L, 700)
        collision = rng.choice((0, 1))  # BGK stays stable at a higher viscosity only
        c = _shear("", L, 0.1 if collision else rng.choice((0.1, 0.2)), 1.0e3 if collision else 1.0e4, collision,
                   rng.randint(10, 50), build)
    elif kind == "batch":
        build = rng.choices(("f32", "f64"), (5, 1))[0]
        n = rng.randint(2, 16)
        if rng.random() < 0.5:
            Ds = [rng.choice((40, 64, 96, 128) if build == "f32" else (16, 24, 32)) for _ in range(n)]
            c = _batch("", ",".join(map(str, Ds)), 12, 6, 2, rng.randint(4, 20) if build == "f32" else rng.randint(2, 6),
                       build)
        else:
            D = rng.choice((15, 20, 30) if build == "f32" else (12, 15))
            c = _batch("", ",".join([str(D)] * n), 45, 20, 3, rng.randint(4, 20) if build == "f32" else 3, build)
    else:
        build = rng.choices(("f32", "f16s", "f64pop", "f64"), (12, 2, 1, 3))[0] if kind == "step" else \
            rng.choices(("f32", "f64"), (3, 1))[0]
        top = 2048 if build in ("f32", "f16s", "f64pop") else 512
        if kind == "adjoint":
            top = 400 if build == "f32" else 128
        ny = int(_log(rng, 64, top))
        nx = max(96, int(ny * rng.uniform(1.5, 2.5)))
        D = float(max(12, int(ny * rng.uniform(0.08, 0.22))))
        nu = _log(rng, 1e-3, 0.03)
        Re, dT = U_IN * D / nu, _log(rng, 0.02, 0.20)
        if kind == "step":
            c = _cyl("", nx, ny, D, Re, dT, rng.randint(1, 40) if build != "f64" else rng.randint(1, 10), build,
                     xf=rng.choice((0.2, 0.25, 0.3)), a_num=rng.choice((2, 3)),
                     psi_mode=rng.choices((0, 1, 2), (8, 1, 1))[0] if build == "f32" else 0)
            # bubbles in flows that stay stable for thousands of passes
            c["boil"] = ny >= 200 and nu >= 4e-3 and c["a_num"] == 2
        else:
            # long enough for the inlet to be heard at the wall
            steps = int(1.25 * (nx * 0.25 - 0.5 * D) / math.sqrt(1.0 / 3.0)) + rng.randint(20, 60)
            c = _adjoint("", nx, ny, D, Re, dT, steps, rng.randint(15, 50), build, boil=False)
    del c["name"]
    return c


# ---------------------------------------------------------------- constants of a run, in FP64 (Sec. II.C, III.D, IV.A)
_COEX = {}


def _coexistence(a, b, R, kappa, Tc, T):
    """Maxwell's equal-area rule for the Peng-Robinson EOS: (rho_v, rho_l) at T."""
    key = (a, b, R, kappa, T)
    if key in _COEX:
        return _COEX[key]
    phi = (1.0 + kappa * (1.0 - math.sqrt(T / Tc))) ** 2
    s2 = math.sqrt(2.0)

    def p(r):
        return r * R * T / (1.0 - b * r) - a * phi * r * r / (1.0 + 2.0 * b * r - b * b * r * r)

    def bisect(f, lo, hi):
        flo = f(lo)
        for _ in range(300):
            mid = 0.5 * (lo + hi)
            if mid <= lo or mid >= hi:
                break
            fm = f(mid)
            if (fm < 0.0) == (flo < 0.0):
                lo, flo = mid, fm
            else:
                hi = mid
        return 0.5 * (lo + hi)

    def dp(r):
        D, x = 1.0 + 2.0 * b * r - b * b * r * r, 1.0 - b * r
        return R * T / (x * x) - a * phi * (2.0 * r * D - r * r * (2.0 * b - 2.0 * b * b * r)) / (D * D)

    grid = (np.arange(4000) + 0.5) / (4000 * b)
    sign = [dp(r) < 0.0 for r in grid]
    turn = [k for k in range(3999) if sign[k] != sign[k + 1]]
    ra, rb = (bisect(dp, grid[k], grid[k + 1]) for k in turn[:2])

    def prim(v):  # antiderivative of p with respect to v = 1 / rho
        return R * T * math.log(v - b) - a * phi / (2.0 * s2 * b) * math.log((v + b - s2 * b) / (v + b + s2 * b))

    def branches(ps):
        return bisect(lambda r: p(r) - ps, 1e-12, ra), bisect(lambda r: p(r) - ps, rb, (1.0 - 1e-12) / b)

    def area(ps):
        rv, rl = branches(ps)
        return prim(1.0 / rv) - prim(1.0 / rl) - ps * (1.0 / rv - 1.0 / rl)

    hi = p(ra)
    _COEX[key] = branches(bisect(area, max(p(rb), 1e-10 * hi) * (1.0 + 1e-13), hi * (1.0 - 1e-13)))
    return _COEX[key]


def _physics(c):
    """Constants of a cylinder or shear-layer case."""
    shear = c["kind"] == "shear"
    a, b, R, acentric, sigma = (2.0 if shear else float(c["a_num"])) / 49.0, 2.0 / 21.0, 1.0, 0.344, 0.38
    kappa = 0.37464 + 1.54226 * acentric - 0.26992 * acentric * acentric
    Tc = 0.0778 * a / (0.4572 * b * R)
    T_sat = 0.86 * Tc
    rv, rl = _coexistence(a, b, R, kappa, Tc, T_sat)
    nu = (c["Ma"] / math.sqrt(3.0) * c["L"] / c["Re"]) if shear else U_IN * c["D"] / c["Re"]
    return SimpleNamespace(a=a, b=b, R=R, kappa=kappa, Tc=Tc, T_sat=T_sat, rv=rv, rl=rl, nu=nu, al=nu / 0.862,
                           av=nu / 1.5, cv=11.0, G=0.0 if shear else -2.0, sigma=0.0 if shear else sigma,
                           g=0.0 if shear else U_IN * U_IN / (16.0 * c["D"]),
                           T_wall=T_sat + (0.0 if shear else c["dT"]) * Tc)


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _initial(c, seed):
    """FP64 [ny][nx] initial fields of a single domain, from the seed: for a cylinder, saturated liquid with
    density noise and, with boil, a superheated layer on the hot wall and vapour bubbles in the wake."""
    dev = _device()
    gen = torch.Generator(device=dev).manual_seed(1000003 * int(seed) + 17)
    ph = _physics(c)
    nx, ny = (c["L"], c["L"]) if c["kind"] == "shear" else (c["nx"], c["ny"])
    noise = torch.rand((ny, nx), generator=gen, device=dev, dtype=torch.float64) * 2e-4 - 1e-4
    if c["kind"] == "shear":
        y, x = torch.meshgrid(torch.arange(ny, device=dev, dtype=torch.float64) / ny,
                              torch.arange(nx, device=dev, dtype=torch.float64) / nx, indexing="ij")
        u0 = c["Ma"] / math.sqrt(3.0)
        ux = torch.where(y <= 0.5, u0 * torch.tanh(80.0 * (y - 0.25)), u0 * torch.tanh(80.0 * (0.75 - y)))
        uy = u0 * 0.05 * torch.sin(2.0 * math.pi * (x + 0.25))
        return {"rho": 1.0 + 0.1 * noise, "ux": ux, "uy": uy}
    rho = ph.rl + noise
    out = {"rho": rho}
    if c["boil"]:
        y, x = torch.meshgrid(torch.arange(ny, device=dev, dtype=torch.float64),
                              torch.arange(nx, device=dev, dtype=torch.float64), indexing="ij")
        xc, yc, r = c["xf"] * nx, 0.5 * ny, 0.5 * c["D"]
        d = torch.sqrt((x - xc) ** 2 + (y - yc) ** 2) - r
        thick = min(max(0.08 * c["D"], 6.0), 12.0)
        liquid = torch.ones_like(d)
        place = torch.rand(18, generator=gen, device=dev, dtype=torch.float64).cpu().tolist()
        for k in range(6):
            rb = min(max(8.0, (0.10 + 0.10 * place[3 * k]) * c["D"]), 14.0)
            xb = xc + 1.2 * c["D"] + rb + place[3 * k + 1] * max(1.0, 0.9 * nx - xc - 1.2 * c["D"] - 2.0 * rb)
            yb = rb + 6.0 + place[3 * k + 2] * max(1.0, ny - 2.0 * rb - 12.0)
            db = torch.sqrt((x - xb) ** 2 + (y - yb) ** 2) - rb
            liquid = torch.minimum(liquid, 0.5 * (1.0 + torch.tanh(db / 2.5)))
        out["rho"] = ph.rv + (ph.rl - ph.rv) * liquid + noise * liquid
        out["T"] = ph.T_sat + (ph.T_wall - ph.T_sat) * torch.exp(-torch.clamp(d, min=0.0) / thick)
    return out


# ---------------------------------------------------------------- prepare and run
def _sim_args(c):
    k = {"f64": c["build"] == "f64", "storage": {"f16s": "f16s", "f64pop": "f64"}.get(c["build"], "f32")}
    if c["kind"] == "shear":
        return dict(nx=c["L"], ny=c["L"], periodic_x=1, superheat_Tc=0.0, G=0.0, sigma=0.0, energy=0, u_in=0.0,
                    nu_l=c["Ma"] / math.sqrt(3.0) * c["L"] / c["Re"], g=0.0, noise_amp=0.0, collision=c["collision"], **k)
    return dict(nx=c["nx"], ny=c["ny"], D=c["D"], xc=c["xf"] * c["nx"], yc=0.5 * c["ny"], superheat_Tc=c["dT"],
                a=c["a_num"] / 49.0, Re=c["Re"], u_in=U_IN, noise_amp=0.0, psi_mode=c["psi_mode"], **k)


def _domains(c, seed):
    """The domains of a batch: superheat log-spaced 0.01 .. 0.25 Tc, Re 300 (30 on the paper's domain)."""
    Ds = [float(d) for d in c["Ds"].split(",")]
    dTs = np.geomspace(0.01, 0.25, len(Ds))
    return [SimpleNamespace(nx=int(c["W"] * D), ny=int(c["H"] * D), D=D, xc=(0.2 if c["a_num"] == 3 else 0.25) * c["W"] * D,
                            yc=0.5 * c["H"] * D, periodic_x=0, walls=0, superheat_Tc=float(dT), rho_s=0.0,
                            a=c["a_num"] / 49.0, Re=30.0 if c["a_num"] == 3 else 300.0, u_in=U_IN, warmup=0,
                            seed=int(seed) * 64 + k + 1, noise_amp=1e-4)
            for k, (D, dT) in enumerate(zip(Ds, dTs))]


def prepare(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        return SimpleNamespace(case=c, batch=Batch(_domains(c, seed), f64=c["build"] == "f64"))
    init = {k: v.cpu().numpy() for k, v in _initial(c, seed).items()}
    return SimpleNamespace(case=c, sim=Sim(init=init, **_sim_args(c)))


def _planes(t, c):
    """Fields of an FP32 context come back as doubles that hold FP32 values: kept as FP32."""
    return t if c["build"] == "f64" else t.to(torch.float32)


def run(state):
    c = state.case
    if c["kind"] == "batch":
        state.batch.step(c["steps"])
        out = []
        for i in range(len(state.batch)):
            d = state.batch.domain(i)
            hf = d.heat_flux()
            f = _planes(d.fields_device(("rho", "ux", "uy", "T"))[0], c)
            out.append({"q": hf["q_mean"], "flow": f[:3], "T": f[3]})
        return out
    if c["kind"] == "adjoint":
        g = state.sim.adjoint_window(c["steps"], c["ckpt"], per_node=True)
        return {"J": g["J"], "superheat": g["superheat"], "u_in": g["u_in"],
                "Tw": g["Tw"] if c["build"] == "f64" else g["Tw"].astype(np.float32)}
    state.sim.step(c["steps"])
    if c["kind"] == "shear":
        f = _planes(state.sim.fields_device(("rho", "ux", "uy"))[0], c)
        return {"rho": f[0], "u": f[1:3]}
    hf = state.sim.heat_flux()
    f = _planes(state.sim.fields_device(("rho", "ux", "uy", "T", "psi"))[0], c)
    return {"q_now": hf["q_now"], "q_mean": hf["q_mean"], "rho": f[0], "u": f[1:3], "T": f[3], "psi": f[4]}


# ---------------------------------------------------------------- the work of a pass
def work(case):
    """Bytes: per step and node the nine populations and T once in and once out (no T for the shear layer), and the
    fields returned once.  Operations: those of the method's equations, counted once per node and step."""
    c = case
    pop = {"f32": 4, "f16s": 2, "f64pop": 8, "f64": 8}[c["build"]]
    es = 8 if c["build"] == "f64" else 4
    if c["kind"] == "shear":
        n = c["L"] * c["L"]
        return {"bytes": n * (18 * pop * c["steps"] + 3 * es), "flops": n * c["steps"] * 190}
    if c["kind"] == "batch":
        n = sum(d.nx * d.ny for d in _domains(c, 0))
        return {"bytes": n * ((18 * pop + 2 * es) * c["steps"] + 4 * es), "flops": n * c["steps"] * 560}
    n = c["nx"] * c["ny"]
    if c["kind"] == "adjoint":
        # forward; the reverse step reads the state it differentiates, and the adjoint state in and out
        return {"bytes": n * c["steps"] * (20 + 10 + 20) * es, "flops": n * c["steps"] * 4 * 560}
    return {"bytes": n * ((18 * pop + 2 * es) * c["steps"] + 5 * es), "flops": n * c["steps"] * 560}


# ---------------------------------------------------------------- the method in 64 bits
CX = (0, 1, -1, 0, 0, 1, -1, 1, -1)
CY = (0, 0, 0, 1, -1, 1, -1, -1, 1)
OPP = (0, 2, 1, 4, 3, 6, 5, 8, 7)
ISO = {1: 4.0 / 21.0, 2: 4.0 / 45.0, 4: 1.0 / 60.0, 5: 2.0 / 315.0, 8: 1.0 / 5040.0}
HALF = [(x, y) for y in range(3) for x in range(-2, 3) if y > 0 or x > 0]


class _Plain:
    """One domain in FP64 torch: fields [ny][nx], periodic in y, open or periodic in x."""

    def __init__(self, ph, nx, ny, D, xc, yc, periodic, collision=0):
        self.ph, self.nx, self.ny, self.periodic, self.bgk = ph, nx, ny, periodic, collision == 1
        dev = _device()
        self.Tw = None
        y, x = torch.meshgrid(torch.arange(ny, device=dev), torch.arange(nx, device=dev), indexing="ij")
        xc, yc = (torch.tensor(v, dtype=torch.float64, device=dev) for v in (xc, yc))
        r = 0.5 * D
        self.solid = ((x - xc) ** 2 + (y - yc) ** 2 <= r * r) if D > 0 else torch.zeros((ny, nx), dtype=torch.bool, device=dev)
        self.inlet = (x == 0) if not periodic else torch.zeros_like(self.solid)
        self.links = []
        near = torch.zeros_like(self.solid)
        flat = y * nx + x
        for i in range(1, 9):
            if D <= 0:
                break
            src = torch.roll(self.solid, (CY[i], CX[i]), (0, 1)) & ~self.solid  # the cylinder stays off the x edges
            ys, xs = y[src], x[src]
            dx, dy = xs - xc, ys - yc
            A = float(CX[i] ** 2 + CY[i] ** 2)
            B = -(dx * CX[i] + dy * CY[i])
            q = (-B - torch.sqrt(B * B - A * (dx * dx + dy * dy - r * r))) / A
            yp, xp = (ys + CY[i]) % ny, xs + CX[i]
            ok = ~self.solid[yp, xp]
            self.links.append((i, flat[src], yp * nx + xp, q, ok))
            near |= src
        self.near = flat[near]
        dx, dy = x[near] - xc, y[near] - yc
        rr = torch.sqrt((dx * dx + dy * dy).double())
        self.normal = (dx / rr, dy / rr)

    # shifted views of a field: f(x + dx, y + dy), the edge column repeated past an open edge
    def pad(self, f):
        f = torch.cat([f[-2:], f, f[:2]], 0)
        lo, hi = (f[:, -2:], f[:, :2]) if self.periodic else (f[:, :1].expand(-1, 2), f[:, -1:].expand(-1, 2))
        return torch.cat([lo, f, hi], 1)

    def at(self, P, dx, dy):
        return P[2 + dy:2 + dy + self.ny, 2 + dx:2 + dx + self.nx]

    def grad(self, f, lap=False, x=True, y=True):
        P = self.pad(f)
        gx, gy, lp = 0.0, 0.0, 0.0
        for ex, ey in HALF:
            w = ISO[ex * ex + ey * ey]
            p, m = self.at(P, ex, ey), self.at(P, -ex, -ey)
            if ex and x:
                gx = gx + (w * ex) * (p - m)
            if ey and y:
                gy = gy + (w * ey) * (p - m)
            if lap:
                lp = lp + w * ((p - f) + (m - f))
        return gx, gy, 2.0 * lp, P

    def feq(self, rho, u, v):
        """Equilibrium of Eq. (equi): the populations whose central moments are (rho, 0, 0, 2 rho/3, 0, ..., rho/9)."""
        z = torch.zeros_like(rho)
        return self.from_central([rho, z, z, 2.0 * rho / 3.0, z, z, z, z, rho / 9.0], rho, u, v)

    def from_central(self, k, rho, u, v):
        k20, k02 = 0.5 * (k[3] + k[4]), 0.5 * (k[3] - k[4])
        k0, k1, k2, k11, k21, k12, k22 = k[0], k[1], k[2], k[5], k[6], k[7], k[8]
        m10, m01 = k1 + u * k0, k2 + v * k0
        m20, m02 = k20 + 2.0 * u * k1 + u * u * k0, k02 + 2.0 * v * k2 + v * v * k0
        m11 = k11 + u * k2 + v * k1 + u * v * k0
        m21 = k21 + v * k20 + 2.0 * u * k11 + u * u * k2 + 2.0 * u * v * k1 + u * u * v * k0
        m12 = k12 + u * k02 + 2.0 * v * k11 + v * v * k1 + 2.0 * u * v * k2 + u * v * v * k0
        m22 = (k22 + 2.0 * u * k12 + 2.0 * v * k21 + v * v * k20 + u * u * k02 + 4.0 * u * v * k11 + 2.0 * u * v * v * k1
               + 2.0 * u * u * v * k2 + u * u * v * v * k0)
        f0 = k0 - m20 - m02 + m22
        e, w = 0.5 * (m10 + m20 - m12 - m22), 0.5 * (-m10 + m20 + m12 - m22)
        n, s = 0.5 * (m01 + m02 - m21 - m22), 0.5 * (-m01 + m02 + m21 - m22)
        ne, sw = 0.25 * (m11 + m21 + m12 + m22), 0.25 * (m11 - m21 - m12 + m22)
        se, nw = 0.25 * (-m11 - m21 + m12 + m22), 0.25 * (-m11 + m21 - m12 + m22)
        return [f0, e, w, n, s, ne, sw, se, nw]

    def start(self, rho, ux, uy, T):
        rho = torch.where(self.solid, self.ph.rl, rho)
        ux, uy = torch.where(self.solid, 0.0, ux), torch.where(self.solid, 0.0, uy)
        f = self.feq(rho, ux, uy)
        return f, torch.where(self.solid, self.ph.T_wall, T), [f[i][:, -1] for i in (2, 6, 8)]

    def pull(self, f, side, u_in):
        U = U_IN
        flats = [g.reshape(-1) for g in f]
        out = []
        for i in range(9):
            if self.periodic:
                v = torch.roll(f[i], (CY[i], CX[i]), (0, 1))
            else:
                v = torch.roll(f[i], CY[i], 0)
                edge = torch.zeros_like(v[:, :1])
                v = torch.cat([edge, v[:, :-1]], 1) if CX[i] == 1 else torch.cat([v[:, 1:], edge], 1) if CX[i] == -1 else v
            out.append(v)
        for i, node, ahead, q, ok in self.links:
            a, b, c = flats[OPP[i]][node], flats[OPP[i]][ahead], flats[i][node]
            v = torch.where(q < 0.5, torch.where(ok, 2.0 * q * a + (1.0 - 2.0 * q) * b, a),
                            a / (2.0 * q) + (2.0 * q - 1.0) / (2.0 * q) * c)
            out[i] = out[i].reshape(-1).index_put((node,), v).reshape(self.ny, self.nx)
        if self.periodic:
            return out, side
        c0 = [g[:, 0] for g in out]
        rho = (c0[0] + c0[3] + c0[4] + 2.0 * (c0[2] + c0[6] + c0[8])) / (1.0 - u_in)
        new = {1: c0[2] + 2.0 / 3.0 * rho * u_in, 5: c0[6] - 0.5 * (c0[3] - c0[4]) + rho * u_in / 6.0,
               7: c0[8] + 0.5 * (c0[3] - c0[4]) + rho * u_in / 6.0}
        for i, v in new.items():
            out[i] = torch.cat([v[:, None], out[i][:, 1:]], 1)
        after = []
        for s, i in zip(side, (2, 6, 8)):
            v = (s + U * torch.roll(f[i][:, -1], CY[i], 0)) / (1.0 + U)
            out[i] = torch.cat([out[i][:, :-1], v[:, None]], 1)
            after.append(v)
        return out, after

    def rhs(self, T, fz):
        ph = self.ph
        gx, gy, lap, P = self.grad(T, lap=True)

        def up(v, sh):
            return torch.where(v >= 0.0, sh(-2) - 6.0 * sh(-1) + 2.0 * sh(1), -2.0 * sh(-1) + 6.0 * sh(1) - sh(2)) / 6.0

        conv = (fz.ux * up(fz.ux, lambda k: self.at(P, k, 0) - T) + fz.uy * up(fz.uy, lambda k: self.at(P, 0, k) - T))
        s = 1.0 + ph.kappa * (1.0 - torch.sqrt(T / ph.Tc))
        dpdT = fz.rep - fz.att * (-ph.kappa * s / torch.sqrt(T * ph.Tc))
        return -conv + (fz.lam * lap + fz.lx * gx + fz.ly * gy - T * dpdT * fz.divu) / (fz.rho * ph.cv)

    def step(self, f, T, side, u_in, Tw, energy):
        ph = self.ph
        f, side = self.pull(f, side, u_in)
        rho = sum(f[1:], f[0])
        rho = torch.where(self.solid, ph.rl, rho)
        zero = torch.zeros_like(rho)
        psi, Fmx, Fmy = zero, zero, zero
        if ph.G != 0.0:
            s = 1.0 + ph.kappa * (1.0 - torch.sqrt(T / ph.Tc))
            p = rho * ph.R * T / (1.0 - ph.b * rho) - ph.a * s * s * rho * rho / (1.0 + 2.0 * ph.b * rho - (ph.b * rho) ** 2)
            psi = torch.sqrt(2.0 * (p - rho / 3.0) / (ph.G / 3.0))
            gx, gy, _, _ = self.grad(psi)
            Fmx, Fmy = -ph.G / 3.0 * psi * gx, -ph.G / 3.0 * psi * gy
        Fx, Fy = Fmx - (rho - ph.rl) * ph.g, Fmy
        w = torch.clamp((rho - ph.rv) / (ph.rl - ph.rv), 0.0, 1.0)
        omega = 1.0 / (3.0 * ph.nu + 0.5)  # nu_l = nu_v
        m1, m2 = f[1] - f[2] + f[5] - f[6] + f[7] - f[8], f[3] - f[4] + f[5] - f[6] - f[7] + f[8]
        ux, uy = (m1 + 0.5 * Fx) / rho, (m2 + 0.5 * Fy) / rho
        if self.bgk:
            cf = 1.0 - 0.5 * omega
            g = self.from_central([omega * rho, cf * Fx, cf * Fy, omega * 2.0 * rho / 3.0, zero, zero, cf * Fy / 3.0,
                                   cf * Fx / 3.0, omega * rho / 9.0], rho, ux, uy)
            g = [(1.0 - omega) * p + q for p, q in zip(f, g)]
        else:
            k4 = f[1] + f[2] - f[3] - f[4] - 2.0 * ux * m1 + 2.0 * uy * m2 + (ux * ux - uy * uy) * rho
            k5 = f[5] + f[6] - f[7] - f[8] - uy * m1 - ux * m2 + ux * uy * rho
            aF = ph.sigma / (psi * psi) * (Fmx * Fmx + Fmy * Fmy) if ph.G != 0.0 else zero
            g = self.from_central([rho, 0.5 * Fx, 0.5 * Fy, 2.0 * rho / 3.0 + 2.0 * aF, (1.0 - omega) * k4,
                                   (1.0 - omega) * k5, Fy / 6.0, Fx / 6.0, rho / 9.0 + 2.0 / 3.0 * aF], rho, ux, uy)
        ux, uy = torch.where(self.solid, 0.0, ux), torch.where(self.solid, 0.0, uy)
        q = zero.sum()
        if energy:
            lam = rho * ph.cv * (ph.av + w * (ph.al - ph.av))
            lx, ly, _, _ = self.grad(lam)
            divu = self.grad(ux, y=False)[0] + self.grad(uy, x=False)[1]
            fz = SimpleNamespace(rho=rho, ux=ux, uy=uy, lam=lam, lx=lx, ly=ly, divu=divu,
                                 rep=rho * ph.R / (1.0 - ph.b * rho),
                                 att=ph.a * rho * rho / (1.0 + 2.0 * ph.b * rho - (ph.b * rho) ** 2))
            if len(self.near):
                gx, gy, _, _ = self.grad(T)
                b = self.near
                q = (-lam.reshape(-1)[b] * (gx.reshape(-1)[b] * self.normal[0] + gy.reshape(-1)[b] * self.normal[1])).mean()

            def fixed(t):
                return torch.where(self.solid, Tw, torch.where(self.inlet, ph.T_sat, t))

            T1 = fixed(T + self.rhs(T, fz))
            T = fixed(0.5 * (T + T1 + self.rhs(T1, fz)))
        return g, T, side, rho, ux, uy, psi, q


def _noise(nx, ny, seed):
    """The library's default density noise: SplitMix64 stream `seed` mapped to [-1, 1)."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + (np.arange(nx * ny, dtype=np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    return torch.from_numpy((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53 * 2.0 - 1.0).reshape(ny, nx).to(_device())


def _march(dom, init, steps, energy):
    f, T, side = dom.start(*init)
    qs = []
    for _ in range(steps):
        f, T, side, rho, ux, uy, psi, q = dom.step(f, T, side, U_IN, dom.ph.T_wall, energy)
        qs.append(q)
    return torch.stack(qs), rho, ux, uy, T, psi


def _full(dom, v):
    return torch.full((dom.ny, dom.nx), v, dtype=torch.float64, device=_device())


def exact(case, seed):
    c = dict(case)
    if c["kind"] == "batch":
        out = []
        for d in _domains(c, seed):
            ph = _physics({"kind": "step", "a_num": c["a_num"], "D": d.D, "Re": d.Re, "dT": d.superheat_Tc})
            dom = _Plain(ph, d.nx, d.ny, d.D, d.xc, d.yc, False)
            rho = ph.rl + d.noise_amp * _noise(d.nx, d.ny, d.seed)
            with torch.no_grad():
                q, rho, ux, uy, T, _ = _march(dom, (rho, _full(dom, U_IN), _full(dom, 0.0), _full(dom, ph.T_sat)), c["steps"],
                                              True)
            out.append({"q": float(q.mean()), "flow": torch.stack([rho, ux, uy]), "T": T})
        return out
    init = _initial(c, seed)
    ph = _physics(c)
    if c["kind"] == "shear":
        dom = _Plain(ph, c["L"], c["L"], 0.0, 0.0, 0.0, True, c["collision"])
        with torch.no_grad():
            _, rho, ux, uy, _, _ = _march(dom, (init["rho"], init["ux"], init["uy"], _full(dom, ph.T_sat)), c["steps"], False)
        return {"rho": rho, "u": torch.stack([ux, uy])}
    dom = _Plain(ph, c["nx"], c["ny"], c["D"], c["xf"] * c["nx"], 0.5 * c["ny"], False)
    full = (init["rho"], _full(dom, U_IN), _full(dom, 0.0), init.get("T", _full(dom, ph.T_sat)))
    if c["kind"] == "step":
        with torch.no_grad():
            q, rho, ux, uy, T, psi = _march(dom, full, c["steps"], True)
        return {"q_now": float(q[-1]), "q_mean": float(q.mean()), "rho": rho, "u": torch.stack([ux, uy]), "T": T, "psi": psi}
    # the window's gradient by reverse-mode differentiation of the plain step
    f, T, side = dom.start(*full)
    Tw = _full(dom, ph.T_wall).requires_grad_(True)
    u_in = torch.tensor(U_IN, dtype=torch.float64, device=Tw.device, requires_grad=True)

    def one(u, tw, T, *fs):
        g, T, s, _, _, _, _, q = dom.step(list(fs[:9]), T, list(fs[9:]), u, tw, True)
        return (T, q, *g, *s)

    T = torch.where(dom.solid, Tw, T)
    total = 0.0
    for _ in range(c["steps"]):
        T, q, *fs = checkpoint(one, u_in, Tw, T, *f, *side, use_reentrant=False)
        f, side = fs[:9], fs[9:]
        total = total + q
    J = total / c["steps"]
    J.backward()
    gw = torch.where(dom.solid, Tw.grad, 0.0)
    return {"J": float(J.detach()), "superheat": float(ph.Tc * gw.sum()), "u_in": float(u_in.grad), "Tw": gw}
