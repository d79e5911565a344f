"""Performance cases of the lattice Boltzmann library: what its users run, at the sizes they run it.

Every case is one whole call sequence of a user's program: set initial fields (device arrays), advance a
number of steps (or run the adjoint over them), read the fields back into device arrays.  A program hands
the fields on in the type its run stores populations in (an FP32 run carries FP32 accuracy, a 16-bit run
16-bit accuracy), so they come back as tensors of that type; FP64 runs return the arrays that the library
filled.
"""
import math

import numpy as np
import torch

from paper_2604_13407_gb300 import inputs as I
from paper_2604_13407_gb300 import lbm

# D2Q9 velocities and weights, in the library's population order
EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WEIGHT = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4

PRECISION = {"f64": lbm.F64, "f32": lbm.F32, "f16": lbm.F16DEV, "bf16": lbm.BF16DEV}
RESULT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}
ELEMENT = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}

# The two equations of state of the named configurations and of the paper's own experiments, with their
# coexistence densities (Maxwell): Carnahan-Starling at 0.7 T_c (liquid to gas about 39), van der Waals at
# T_r = 0.5 (113) and 0.54 (71).  rho_max: a little below the density where psi stops being real.
EOS = {
    "cs": dict(eos=1, a=1.0, b=4.0, R=1.0, K_eos=1.0, T=0.7 * 0.3773 / 4.0, rho_g=0.009291723294794338,
               rho_l=0.3581443962580134, rho_max=0.0),
    "vdw50": dict(eos=0, a=9.0 / 49.0, b=2.0 / 21.0, R=1.0, K_eos=1.0 / 16.0, T=0.28571428571428575,
                  rho_g=0.076113825017658, rho_l=8.604722001225264, rho_max=9.98),
    "vdw54": dict(eos=0, a=9.0 / 49.0, b=2.0 / 21.0, R=1.0, K_eos=1.0 / 16.0, T=0.3085714285714286,
                  rho_g=0.11878472576668407, rho_l=8.407408147289528, rho_max=9.94),
}
EPSILON = {"cs": 1.895, "vdw50": 1.895, "vdw54": 2.0}


def listed():
    return [
        # a small two-phase channel of odd size, original scheme: the smallest lattices, where a step is
        # little but latency (parameter studies, tests)
        dict(name="ragged_37x23_f32", kind="slab", nx=37, ny=23, prec="f32", eos="cs", scheme=0, walls="y", steps=100),
        # the library's default parameters: the grid-aligned two-phase Poiseuille channel in FP64, a column
        # that is stepped 20k times and more
        dict(name="channel_4x128_f64", kind="slab", nx=4, ny=128, prec="f64", eos="cs", scheme=1, walls="y", steps=100),
        # the grid-oblique two-phase channel of the paper's Table 1, FP64, half-way walls on solid bands
        dict(name="oblique_256_f64", kind="bands", nx=256, ny=256, prec="f64", eos="vdw54", scheme=1, walls="", steps=20),
        # FP64 spinodal decomposition: the accuracy reference of the throughput workload
        dict(name="spinodal_1024_f64", kind="spinodal", nx=1024, ny=1024, prec="f64", eos="cs", scheme=1, walls="", steps=4),
        # the paper's droplet falling in a vertical channel (Sec. 3.3): sampled every few steps for U_c
        dict(name="fall_256x2048_f32", kind="drop", nx=256, ny=2048, prec="f32", eos="vdw50", scheme=1, walls="x", steps=40, diagnostics=True),
        # the paper's annular shear flow (Sec. 3.2): odd lattice, half-way cylinders, force field, wall densities
        dict(name="annular_517_f32", kind="annular", nx=517, ny=517, prec="f32", eos="vdw50", scheme=1, walls="", steps=40),
        # annular shear between a resting and a moving cylinder, interpolated moving walls
        dict(name="annulus_1024_f32", kind="annulus", nx=1024, ny=1024, prec="f32", eos="cs", scheme=1, walls="", steps=40),
        # the grid-oblique channel with a viscosity ratio of ten
        dict(name="oblique_512_f32", kind="bands", nx=512, ny=512, prec="f32", eos="cs", scheme=1, walls="", tau_l=1.0, tau_g=0.55, steps=40),
        # droplet falling in the long channel, populations stored in FP16
        dict(name="fall_512x4096_f16", kind="drop", nx=512, ny=4096, prec="f16", eos="cs", scheme=1, walls="x", steps=20),
        # the throughput headline: periodic spinodal decomposition in FP32
        dict(name="spinodal_8192_f32", kind="spinodal", nx=8192, ny=8192, prec="f32", eos="cs", scheme=1, walls="", tau_l=1.0, tau_g=1.0, steps=20),
        # gradient of the time-averaged wall force of a droplet channel: the adjoint workload, and at a size
        # whose states exceed the L2 cache
        dict(name="adjoint_256x1024_f32", kind="adjoint", nx=256, ny=1024, prec="f32", eos="cs", scheme=1, walls="x", steps=60, every=20),
        dict(name="adjoint_2048_f32", kind="adjoint", nx=2048, ny=2048, prec="f32", eos="cs", scheme=1, walls="x", steps=24, every=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("spinodal", "spinodal", "slab", "slab", "drop", "bands", "annulus", "annular", "adjoint"))
    prec = rng.choice(("f64", "f32", "f32", "f16", "bf16"))
    eos = rng.choice(("cs", "cs", "vdw50"))
    walls = {"spinodal": ("",), "slab": ("y",), "drop": ("x", "", "xy"), "adjoint": ("x", "y", "xy")}.get(kind, ("",))
    case = dict(kind=kind, prec=prec, eos=eos, scheme=rng.choice((0, 1, 1)), walls=rng.choice(walls))
    top = 1 << (18 if prec == "f64" else 22)  # nodes
    if kind in ("bands", "annulus", "annular"):
        n = _log(rng, 48, 400 if prec == "f64" else 1600)
        case.update(nx=n, ny=n)
    elif kind == "slab":
        case.update(nx=_log(rng, 4, 512), ny=_log(rng, 16, 512))
    else:
        nx = _log(rng, 24, 4096 if kind == "spinodal" else 1024)
        ny = _log(rng, 24, 4096)
        case.update(nx=nx, ny=max(24, min(ny, top // nx)))
    if kind == "adjoint":
        case.update(eos="cs", ny=min(case["ny"], (1 << (16 if prec == "f64" else 20)) // case["nx"]))
    if case["walls"] != "" and rng.random() < 0.5 and kind != "adjoint":
        case.update(tau_l=1.0, tau_g=0.7)
    nodes = case["nx"] * case["ny"]
    case["steps"] = max(4, min(100, (1 << (20 if prec == "f64" else 25)) // nodes))
    if kind == "adjoint":
        case["steps"] = max(4, min(60, case["steps"] // 2))
        case["every"] = rng.choice((1, 3, max(1, case["steps"] // 3), case["steps"]))
    if kind in ("drop", "slab"):
        case["diagnostics"] = rng.random() < 0.4
    return case


# ------------------------------------------------------------------ inputs ---

def _params(case):
    e = EOS[case["eos"]]
    k = -EPSILON[case["eos"]] / 16.0
    kind, prec = case["kind"], case["prec"]
    g = {}
    if kind in ("slab", "bands"):
        f = 1e-7 if kind == "slab" else 4e-9
        g = dict(Fx=f) if kind == "slab" else dict(Fx=f / math.sqrt(2.0), Fy=f / math.sqrt(2.0))
    elif kind in ("drop", "adjoint"):
        g = dict(force_mode=lbm.FORCE_BUOYANT, Fy=-2e-6)
    elif kind == "annular":
        g = dict(force_mode=lbm.FORCE_FIELD)
    half = prec in ("f16", "bf16")
    return dict(nx=case["nx"], ny=case["ny"], periodic_x=int("x" not in case["walls"]),
                periodic_y=int("y" not in case["walls"]), precision=PRECISION[prec], scheme=case["scheme"],
                k1=k, k2=k, tau_l=case.get("tau_l", 0.8), tau_g=case.get("tau_g", 0.8), rho_s=e["rho_g"],
                rho_ref=e["rho_g"], per_node_ref=int(half),
                storage_scale_log2=(18 if case["eos"] == "cs" else 14) if prec == "f16" else 0, **e, **g)


def _grid(case):
    y, x = np.mgrid[0:case["ny"], 0:case["nx"]].astype(np.float64)
    return x, y


def _crossing(px, py, dx, dy, r):
    """Smallest t in (0, 1] with |p + t d| = r (nan where there is none)."""
    a, b, c = dx * dx + dy * dy, 2.0 * (px * dx + py * dy), px * px + py * py - r * r
    s = np.sqrt(b * b - 4.0 * a * c)
    t0, t1 = (-b - s) / (2.0 * a), (-b + s) / (2.0 * a)
    inside = lambda t: (t > 1e-12) & (t <= 1.0 + 1e-12)  # noqa: E731
    return np.where(inside(t0), t0, np.where(inside(t1), t1, np.nan))


def _geometry(case):
    """solid, wall_u, q, force_field, wall_rho (host arrays or None)."""
    kind, nx, ny = case["kind"], case["nx"], case["ny"]
    if kind == "bands":
        return I.oblique_band_walls(nx), None, None, None, None
    if kind not in ("annulus", "annular"):
        return (None,) * 5
    e = EOS[case["eos"]]
    x, y = _grid(case)
    x -= (nx - 1) / 2.0
    y -= (ny - 1) / 2.0
    r = np.hypot(x, y)
    r_in, r_out = 0.125 * nx, 0.47 * nx
    solid = ((r <= r_in) | (r >= r_out)).astype(np.uint8)
    turn = np.stack([-y, x]) / np.where(r > 0, r, 1.0)
    if kind == "annular":
        field = 3e-6 * (r / r_out) ** 2 * turn * (solid == 0)
        return solid, None, None, field, np.where(r <= r_in, e["rho_g"], e["rho_l"])
    wall_u = 0.01 * turn * (r >= r_out)
    q = np.full((8, ny, nx), 0.5)
    with np.errstate(invalid="ignore"):
        for d in range(1, 9):
            ahead = np.roll(solid, (-EY[d], -EX[d]), (0, 1)).astype(bool)
            inner = np.roll(r <= r_in, (-EY[d], -EX[d]), (0, 1))
            at = ahead & (solid == 0)
            t = _crossing(x, y, EX[d], EY[d], np.where(inner, r_in, r_out))
            q[d - 1] = np.where(at & np.isfinite(t), np.clip(t, 1e-3, 1.0), 0.5)
    return solid, wall_u, q, None, None


def _fields(case, seed):
    """Initial rho, ux, uy (float64, on the GPU): the phases of the set-up with their place jittered by the
    seed, and a smooth random velocity (a drift and a few Fourier modes, |u| up to about 0.1; 0.04 at the larger
    density ratios), at rest on solid nodes."""
    e = EOS[case["eos"]]
    nx, ny, kind = case["nx"], case["ny"], case["kind"]
    dev = torch.device("cuda")
    g = torch.Generator().manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
    jx, jy = (torch.rand(2, generator=g, dtype=torch.float64) * 2 - 1).tolist()
    x = torch.arange(nx, dtype=torch.float64, device=dev)[None, :]
    y = torch.arange(ny, dtype=torch.float64, device=dev)[:, None]
    rl, rg = e["rho_l"], e["rho_g"]

    def layer(d, width):  # 1 inside |d| < width / 2, tanh edges of width 4
        return 0.5 * (torch.tanh(0.5 * (d + width / 2.0)) - torch.tanh(0.5 * (d - width / 2.0)))

    if kind == "spinodal":
        gd = torch.Generator(device=dev).manual_seed(int(seed) & 0x7FFFFFFFFFFFFFFF)
        noise = torch.rand((ny, nx), generator=gd, dtype=torch.float64, device=dev) * 2 - 1
        rho = 0.5 * (rl + rg) * (1.0 + 0.01 * noise)
    else:
        if kind == "slab":
            c = layer(y - (ny - 1) / 2.0 - jy, ny / 2.0).expand(ny, nx)
        elif kind == "bands":
            c = layer(torch.remainder(x - y, nx) - (nx - 1) / 2.0 - jy, nx / 2.0)
        elif kind in ("annulus", "annular"):
            r = torch.hypot(x - (nx - 1) / 2.0, y - (ny - 1) / 2.0)
            c = layer(r - (0.25 * nx + jx), 0.12 * nx) if kind == "annulus" else 0.5 + 0.5 * torch.tanh(0.5 * (r - 0.2 * nx - jx))
        else:
            radius = max(5.0, min(0.3 * min(nx, ny), 64.0))
            dx = torch.remainder(x - (nx / 2.0 + 2 * jx) + nx / 2.0, nx) - nx / 2.0
            dy = torch.remainder(y - (0.6 * ny + 2 * jy) + ny / 2.0, ny) - ny / 2.0
            c = 0.5 - 0.5 * torch.tanh(0.5 * (torch.hypot(dx, dy) - radius))
        rho = rg + (rl - rg) * c
    amp = 0.05 if case["eos"] == "cs" and case.get("tau_g", 0.8) >= 0.7 else 0.02
    u = []
    for k in range(2):
        a = torch.rand(6, generator=g, dtype=torch.float64) * 2 * math.pi
        a = a.tolist()
        s = sum(torch.cos(2 * math.pi * ((1 + m) * x / nx + (m % 2) * y / ny) + a[2 * m]) * torch.cos(2 * math.pi * (1 + m) * y / ny + a[2 * m + 1])
                for m in range(3)) / 3.0
        u.append(amp * (s + (-0.5 if k == 1 and kind in ("drop", "adjoint") else 0.5)))
    return rho.contiguous(), u[0].contiguous(), u[1].contiguous()


def prepare(case, seed):
    solid, wall_u, q, field, wall_rho = _geometry(case)
    sim = lbm.Simulation(lbm.default_params(**_params(case)), stream=torch.cuda.current_stream())
    if solid is not None:
        sim.set_geometry(solid, wall_u, q, field)
    if wall_rho is not None:
        sim.set_wall_density(wall_rho)
    rho, ux, uy = _fields(case, seed)
    if solid is not None:
        still = torch.from_numpy(solid).to(rho.device) == 0
        e = EOS[case["eos"]]
        rho = torch.where(still, rho, torch.full_like(rho, e["rho_g"]))
        ux, uy = ux * still, uy * still
    out = tuple(torch.empty_like(rho) for _ in range(3))
    return dict(case=case, sim=sim, fields=(rho, ux, uy), out=out)


def run(state):
    case, sim = state["case"], state["sim"]
    sim.init_fields(*state["fields"])
    got = {}
    if case["kind"] == "adjoint":
        J, grad, _ = sim.adjoint(case["steps"], case["every"], lbm.OBJ_WALL_FORCE_Y)
        got["J"] = J
        got["grad"] = torch.as_tensor(grad, dtype=RESULT["f64" if case["prec"] == "f64" else "f32"])
    else:
        sim.step(case["steps"])
    if case.get("diagnostics"):
        d = sim.diagnostics()
        got["mass"], got["u_max"] = float(d[0]), float(d[9])
        got["U_c"] = float(d[7] / d[8])
    sim.moments(out=state["out"])
    got["rho"], got["ux"], got["uy"] = (a.to(RESULT[case["prec"]]) for a in state["out"])
    return got


def work(case):
    nodes, steps, b = case["nx"] * case["ny"], case["steps"], ELEMENT[case["prec"]]
    step = 18 * b + (8 if b == 2 else 0)  # every population read and written once (16-bit: and the reference density)
    size = nodes * (steps * step + 24 + 3 * b)
    flops = nodes * steps * 250
    if case["kind"] == "adjoint":  # and backwards: the state and the adjoint state read, the adjoint state written
        real = 8 if b == 8 else 4
        size += nodes * steps * (step // 2 + 18 * real)
        flops += nodes * steps * 750
    return {"bytes": size, "flops": flops}


# ------------------------------------------------------- plain FP64 step ------

_M = ((1, 1, 1, 1, 1, 1, 1, 1, 1), (-4, -1, -1, -1, -1, 2, 2, 2, 2), (4, -2, -2, -2, -2, 1, 1, 1, 1),
      (0, 1, 0, -1, 0, 1, -1, -1, 1), (0, -2, 0, 2, 0, 1, -1, -1, 1), (0, 0, 1, 0, -1, 1, 1, -1, -1),
      (0, 0, -2, 0, 2, 1, 1, -1, -1), (0, 1, -1, 1, -1, 0, 0, 0, 0), (0, 0, 0, 0, 0, 1, -1, 1, -1))


class _Plain:
    """The step in FP64 torch operations over whole fields."""

    def __init__(self, case, dev):
        self.p = p = _params(case)
        nx, ny = case["nx"], case["ny"]
        solid, wall_u, q, field, wall_rho = _geometry(case)
        t = lambda a: None if a is None else torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
        self.solid = torch.zeros((ny, nx), dtype=torch.bool, device=dev) if solid is None else t(solid).bool()
        self.any_solid = solid is not None
        self.wall_u, self.q, self.field, self.wall_rho = t(wall_u), t(q), t(field), t(wall_rho)
        self.M = torch.tensor(_M, dtype=torch.float64, device=dev)
        self.inv = (self.M / (self.M * self.M).sum(1, keepdim=True)).T.contiguous()
        xs, ys = torch.arange(nx, device=dev)[None, :], torch.arange(ny, device=dev)[:, None]
        self.beyond, self.wall = [], []
        for i in range(9):  # x + e_i beyond a non-periodic edge; and a wall of either kind
            o = torch.zeros((ny, nx), dtype=torch.bool, device=dev)
            if not p["periodic_x"]:
                o = o | (xs + EX[i] < 0) | (xs + EX[i] >= nx)
            if not p["periodic_y"]:
                o = o | (ys + EY[i] < 0) | (ys + EY[i] >= ny)
            self.beyond.append(o)
            self.wall.append(o | self.ahead(self.solid, i))

    @staticmethod
    def ahead(a, i):  # a(x + e_i)
        return torch.roll(a, (-EY[i], -EX[i]), (0, 1)) if i else a

    def psi(self, rho, G, T):
        p = self.p
        if p["eos"] == 0:
            pe = p["K_eos"] * (rho * p["R"] * T / (1 - p["b"] * rho) - p["a"] * rho * rho)
        else:
            h = p["b"] * rho / 4
            pe = p["K_eos"] * (rho * p["R"] * T * (1 + h + h * h - h ** 3) / (1 - h) ** 3 - p["a"] * rho * rho)
        return torch.sqrt(2 * (pe - rho / 3) / G)

    def pull(self, A):
        f = []
        for i in range(9):
            s = self.ahead(A[i], OPP[i])
            if i:
                s = torch.where(self.wall[OPP[i]], self.bounce(A, i), s)
            f.append(s)
        return torch.stack(f)

    def bounce(self, A, i):
        o = OPP[i]
        if self.wall_u is None and self.q is None:
            return A[o]
        mw = 0.0
        if self.wall_u is not None:
            ux, uy = self.ahead(self.wall_u[0], o), self.ahead(self.wall_u[1], o)
            mw = 6 * WEIGHT[o] * A.sum(0) * (EX[i] * ux + EY[i] * uy)
        q = torch.full_like(A[0], 0.5) if self.q is None else self.q[o - 1]
        q = torch.where((q < 0.5) & self.wall[i], torch.full_like(q, 0.5), q)
        near = 2 * q * A[o] + (1 - 2 * q) * self.ahead(A[o], i) + mw
        far = A[o] / (2 * q) + (2 * q - 1) / (2 * q) * A[i] + mw / (2 * q)
        return torch.where(q < 0.5, near, torch.where(q == 0.5, A[o] + mw, far))

    def macro(self, A, th):
        """Pulled populations, rho, S, psi, total force and velocity of the state A; th = (Fx, Fy, G, T)."""
        p = self.p
        f = self.pull(A)
        rho = f.sum(0)
        if self.any_solid:
            rho = torch.where(self.solid, torch.full_like(rho, p["rho_s"]) if self.wall_rho is None else self.wall_rho, rho)
        psi = self.psi(rho, th[2], th[3])
        psi_s = self.psi(torch.full_like(rho[0, 0], p["rho_s"]), th[2], th[3])
        S = [0.0, 0.0]
        for i in range(1, 9):
            v = torch.where(self.beyond[i], psi_s, self.ahead(psi, i)) * (1 / 3 if i <= 4 else 1 / 12)
            S = [S[0] + EX[i] * v, S[1] + EY[i] * v]
        mode = p.get("force_mode", 0)
        if mode == 2:
            ext = self.field
        else:
            ext = [th[k] * (rho - p["rho_g"]) if mode == 1 else th[k] for k in (0, 1)]
        F = [-th[2] * psi * S[k] + ext[k] for k in (0, 1)]
        j = [(f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7]), (f[2] - f[4]) + (f[5] + f[6]) - (f[7] + f[8])]
        u = [(j[k] + 0.5 * F[k]) / rho for k in (0, 1)]
        return f, rho, S, F, u

    def equilibrium(self, rho, ux, uy):
        u2, d = ux * ux + uy * uy, ux * ux - uy * uy
        return [rho, rho * (3 * u2 - 2), rho * (1 - 3 * u2), rho * ux, -rho * ux, rho * uy, -rho * uy, rho * d, rho * ux * uy]

    def back(self, m):
        m = torch.stack(m)
        return (self.inv @ m.reshape(9, -1)).reshape(m.shape)

    def step(self, A, th):
        p = self.p
        f, rho, S, F, (ux, uy) = self.macro(A, th)
        m = (self.M @ f.reshape(9, -1)).reshape(f.shape)
        meq = self.equilibrium(rho, ux, uy)
        Fu = F[0] * ux + F[1] * uy
        Fm = [0.0, 6 * Fu, -6 * Fu, F[0], -F[0], F[1], -F[1], 2 * (F[0] * ux - F[1] * uy), F[0] * uy + F[1] * ux]
        k1, k2, G = p["k1"], p["k2"], th[2]
        eps = -8 * (k1 + k2)
        X, Y = G * S[0] * S[0], G * S[1] * S[1]
        Q = [0.0] * 9
        Q[1] = 3 * (k1 + 2 * k2) * (X + Y)
        Q[7], Q[8] = k1 * (X - Y), k1 * G * S[0] * S[1]
        Q[2] = -Q[1]
        if p["scheme"] == 1:
            Q[2] = -Q[1] / 2
            Q[4] = ((30 * eps - 15) / 16 * X - 3 * eps / 8 * Y) * ux
            Q[6] = ((30 * eps - 15) / 16 * Y - 3 * eps / 8 * X) * uy
        tau = p["tau_l"]
        if p["tau_l"] != p["tau_g"]:
            w = ((rho - p["rho_g"]) / (p["rho_l"] - p["rho_g"])).clamp(0, 1)
            tau = p["tau_g"] + w * (p["tau_l"] - p["tau_g"])
        sp, sq = 1 / tau, 1 / (0.5 + (1 / 12) / (tau - 0.5))
        s = (1.0, sp, sp, 1.0, sq, 1.0, sq, sp, sp)
        out = self.back([m[k] + Fm[k] - s[k] * (m[k] - meq[k] + 0.5 * Fm[k]) + s[k] * Q[k] for k in range(9)])
        return torch.where(self.solid, A, out) if self.any_solid else out

    def wall_force_y(self, A):
        J = 0.0
        for i in range(1, 9):
            if EY[i]:
                J = J + 2 * EY[i] * torch.where(self.wall[i] & ~self.solid, A[i], torch.zeros_like(A[i])).sum()
        return J


def exact(case, seed):
    dev = torch.device("cuda")
    P = _Plain(case, dev)
    p = P.p
    rho, ux, uy = _fields(case, seed)
    if P.any_solid:
        still = ~P.solid
        rho, ux, uy = torch.where(still, rho, torch.full_like(rho, p["rho_g"])), ux * still, uy * still
    th = torch.tensor([p.get("Fx", 0.0), p.get("Fy", 0.0), -1.0, p["T"]], dtype=torch.float64, device=dev)
    A = P.back(P.equilibrium(rho, ux, uy))
    del rho, ux, uy
    got = {}
    if case["kind"] == "adjoint":
        from torch.utils.checkpoint import checkpoint
        th.requires_grad_(True)
        J = 0.0
        for _ in range(case["steps"]):
            A = checkpoint(P.step, A, th, use_reentrant=False)
            J = J + P.wall_force_y(A) / case["steps"]
        got["grad"] = torch.autograd.grad(J, th)[0].cpu()
        got["J"] = float(J)
        A, th = A.detach(), th.detach()
    else:
        with torch.no_grad():
            for _ in range(case["steps"]):
                A = P.step(A, th)
    with torch.no_grad():
        _, rho, _, _, (ux, uy) = P.macro(A, th)
        fluid = ~P.solid
        ux, uy = ux * fluid, uy * fluid
        if case.get("diagnostics"):
            r = rho[fluid]
            liquid = fluid & (rho > 0.5 * (p["rho_l"] + p["rho_g"]))
            got["mass"], got["u_max"] = float(r.sum()), float(torch.hypot(ux, uy).max())
            got["U_c"] = float((rho * uy)[liquid].sum() / rho[liquid].sum())
    got["rho"], got["ux"], got["uy"] = rho, ux, uy
    return got
