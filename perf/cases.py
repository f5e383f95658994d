"""Performance cases of the thermal cascaded LBM: what a program that uses this package has it do.

A case is a dict of plain values.  `kind` says which calls a pass makes:

    flow     a simulation on a handle the program keeps: set the fields, advance `steps` time
             steps, read rho, u, T back (and the FP64 sums where `sums` is set), with fields
             in device memory or, `host` set, in host arrays
    restart  populations into the handle from device memory, some steps, the FP64 sums against
             a velocity snapshot, populations out again
    batch    many lattices of different sizes advanced together, one launch per step
    serve    requests of different kinds and sizes served to completion

The rest of the dict describes the problem: lattice size, walls, storage format, collision
variant.  Every pass starts from the same fields, so it returns the same outputs each time.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1610_07114_gb300 import serve, tclbm
from paper_1610_07114_gb300 import workloads as W

FIELDS = ("rho", "ux", "uy", "T")


def listed():
    return [
        # the thermal Couette lattice of the paper's heating tests: a few hundred nodes, so a
        # time step is all latency; read out every few hundred steps while it settles
        {"name": "couette_8x64", "kind": "flow", "flow": "couette", "nx": 8, "ny": 64, "steps": 200},
        # the paper's Taylor-Green accuracy lattice: athermal, periodic, small
        {"name": "taylor_green_64", "kind": "flow", "flow": "taylor_green", "nx": 64, "ny": 64, "steps": 500},
        # the shock tube: long and four rows high, equilibrium ends, walls on the x axis
        {"name": "shock_4096x4", "kind": "flow", "flow": "shock", "nx": 4096, "ny": 4, "steps": 500},
        # Rayleigh-Benard on the benchmark's lattice, end to end: host fields in, a chunk of
        # 1000 steps with the Nusselt sum, host fields out
        {"name": "rb_256x128_host", "kind": "flow", "flow": "rb", "nx": 256, "ny": 128, "steps": 1000,
         "host": True, "sums": True},
        # the athermal solver on a lattice of a quarter million nodes (half the populations)
        {"name": "taylor_green_512", "kind": "flow", "flow": "taylor_green", "nx": 512, "ny": 512, "steps": 500},
        # a middle-sized layer in the storage format of the sweep and the server: FP16
        # deviations with stochastic rounding
        {"name": "rb_1024x512_fp16sr", "kind": "flow", "flow": "rb", "nx": 1024, "ny": 512, "steps": 200,
         "storage": "fp16", "rounding": "stochastic"},
        # an odd-sized lattice above the small-lattice range, walls on the x axis by
        # extrapolation, bfloat16 deviations
        {"name": "ragged_2051x1537_bf16", "kind": "flow", "flow": "random", "nx": 2051, "ny": 1537, "steps": 70,
         "walls": "x_nee", "storage": "bf16", "rounding": "nearest"},
        # the large layer in full precision: the memory-bound case
        {"name": "rb_4096x2048_fp32", "kind": "flow", "flow": "rb", "nx": 4096, "ny": 2048, "steps": 100,
         "sums": True},
        # the same layer as the server stores it
        {"name": "rb_4096x2048_fp16sr", "kind": "flow", "flow": "rb", "nx": 4096, "ny": 2048, "steps": 100,
         "storage": "fp16", "rounding": "stochastic"},
        # checkpoint and resume of a medium lattice with a residual check in between
        {"name": "restart_2048x1024", "kind": "restart", "flow": "random", "nx": 2048, "ny": 1024, "steps": 20,
         "walls": "y_zouhe"},
        # the Rayleigh-number sweep: lattices of five sizes advanced together
        {"name": "sweep_48", "kind": "batch", "count": 48, "steps": 64, "storage": "fp16", "rounding": "stochastic"},
        # a burst of mixed requests at the server
        {"name": "serve_16", "kind": "serve", "count": 16, "storage": "fp16", "rounding": "stochastic"},
    ]


WALLS = ("none", "y_zouhe", "y_nee", "x_nee", "x_zouhe", "x_equilibrium", "y_equilibrium")
FORMATS = (("fp32", "nearest"), ("fp32", "nearest"), ("fp16", "stochastic"), ("fp16", "nearest"),
           ("bf16", "nearest"), ("bf16", "stochastic"))


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("flow", "flow", "flow", "flow", "flow", "restart", "batch"))
    storage, rounding = rng.choice(FORMATS)
    if kind == "batch":
        return {"kind": "batch", "count": _log(rng, 2, 48), "steps": _log(rng, 1, 64), "storage": storage,
                "rounding": rounding}
    nodes = _log(rng, 512, 1 << 23)
    aspect = math.exp(rng.uniform(math.log(0.25), math.log(4.0)))
    nx = max(3, int(round(math.sqrt(nodes * aspect))))
    ny = max(3, int(nodes / nx))
    if rng.random() < 0.5:  # half of them on multiples of 32, as most programs choose
        nx, ny = max(32, nx // 32 * 32), max(4, ny // 4 * 4)
    most = min(1000, max(1, int(1.0e9 / (nx * ny) * 0.6)))
    steps = _log(rng, 1, most)
    if kind == "restart":
        nx, ny = min(nx, 2048), min(ny, 1024)
        return {"kind": "restart", "flow": "random", "nx": nx, "ny": ny, "steps": min(steps, 50),
                "walls": rng.choice(WALLS), "storage": storage, "rounding": rounding}
    flow = rng.choice(("rb", "rb", "couette", "taylor_green", "shock", "random", "random", "random"))
    case = {"kind": "flow", "flow": flow, "nx": nx, "ny": ny, "steps": steps, "storage": storage,
            "rounding": rounding, "sums": rng.random() < 0.3, "host": rng.random() < 0.2}
    if flow == "rb":
        case["ny"] = max(16, ny)
    elif flow == "couette":
        case["nx"], case["ny"] = min(nx, 64), min(max(8, ny), 1024)
    elif flow == "taylor_green":
        case["nx"] = case["ny"] = max(8, int(math.sqrt(nx * ny)))
        case["thermal"] = rng.random() < 0.5
    elif flow == "shock":
        case["nx"], case["ny"] = min(max(64, nx * ny // 8), 8192), _log(rng, 4, 64)
    else:
        case["walls"] = rng.choice(WALLS)
        case["steps"] = min(steps, 200)
        case["force"] = rng.choice(("none", "accel", "taylor_green"))
        case["variant"] = rng.choice(("corr", "corr", "corr", "thermal", "athermal"))
        case["visc_law"] = rng.choice(("nu", "nu", "mu", "mu_T", "w1"))
        case["work"] = case["variant"] != "athermal" and rng.random() < 0.25
    return case


# ------------------------------------------------------------------ problems and inputs


def _problem(case):
    """The package's case dict of a case (no fields)."""
    storage, nx, ny = case.get("storage", "fp32"), case["nx"], case["ny"]
    flow = case["flow"]
    if flow == "couette":
        d, _ = W.couette(nx, ny, storage=storage, fields=False)
    elif flow == "taylor_green":
        # u0 of the paper's 64 x 64 lattice, Reynolds number kept as the lattice grows
        nu, u0, k = 0.02, 0.026 * 64.0 / max(nx, 64), 2.0 * math.pi / nx
        d, _ = W.taylor_green(nx, F0=2.0 * nu * k * k * u0, nu=nu, thermal=bool(case.get("thermal")),
                              storage=storage, fields=False)
    elif flow == "shock":
        d, _ = W.shock_tube(64, 4, storage=storage)
        d["nx"], d["ny"] = nx, ny
    elif flow == "rb":
        d, _ = W.rayleigh_benard(nx, ny, Ra=min(1e5, W.rb_max_resolved_ra(ny)), storage=storage, fields=False)
    else:
        variant, force, law = case.get("variant", "corr"), case.get("force", "accel"), case.get("visc_law", "nu")
        visc = {"nu": 0.03, "mu": 0.03, "mu_T": 0.03, "w1": 1.45}[law]
        d = W.base_case(nx, ny, thermal=variant != "athermal", correction=variant == "corr", visc_law=law, visc=visc,
                        w2=1.2, w3=1.1, w4=0.9, storage=storage)
        if force == "accel":
            d["force"] = {"kind": "accel", "ax": 1e-5, "ay": -2e-5, "amp": 0.0}
        elif force == "taylor_green":
            d["force"] = {"kind": "taylor_green", "ax": 0.0, "ay": 0.0, "amp": 1e-5}
        walls = case.get("walls", "none")
        if walls != "none":
            axis, kind = walls.split("_")
            wall = {"kind": kind, "ux": 0.0, "uy": 0.0, "therm": "fixed"}
            moving = {"uy" if axis == "x" else "ux": 0.03} if kind == "zouhe" else {}
            d["walls"][axis + "-"] = dict(wall, T=1.004, rho=1.002)
            d["walls"][axis + "+"] = dict(wall, T=0.996, rho=0.999, **moving)
        d["work"] = bool(case.get("work"))
    d["rounding"] = case.get("rounding", "nearest")
    return d


def _fields(case, seed):
    """Initial rho, u, T as float64 device tensors [ny][nx], from the seed alone."""
    nx, ny, flow = case["nx"], case["ny"], case["flow"]
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    o = dict(dtype=torch.float64, device="cuda")

    def smooth(amp):
        a = torch.rand((ny, nx), generator=g, **o).mul_(2.0).sub_(1.0)
        b = a + a.roll(1, 0) + a.roll(-1, 0) + a.roll(1, 1) + a.roll(-1, 1)
        return b.mul_(amp / 5.0)

    one, zero = torch.ones((ny, nx), **o), torch.zeros((ny, nx), **o)
    x = torch.arange(nx, **o)[None, :]
    y = torch.arange(ny, **o)[:, None]
    if flow == "couette":  # a shear layer on its way to the linear profile, T = 1
        eta = y / (ny - 1)
        uy = 0.01 * torch.sin(math.pi * eta) * torch.sin(2.0 * math.pi * x / nx)
        return {"rho": one + smooth(1e-4), "ux": 0.05 * eta ** 2 + smooth(1e-3), "uy": uy + smooth(1e-4),
                "T": one + smooth(1e-4)}
    if flow == "taylor_green":
        u0, k = 0.026 * 64.0 / max(nx, 64), 2.0 * math.pi / nx
        return {"rho": one + smooth(1e-4), "ux": 0.8 * u0 * torch.sin(k * x) * torch.sin(k * y) + smooth(1e-2 * u0),
                "uy": 0.8 * u0 * torch.cos(k * x) * torch.cos(k * y) + smooth(1e-2 * u0), "T": one + smooth(1e-4)}
    if flow == "shock":
        left = (x < nx // 2).double() * torch.ones_like(y)
        return {"rho": 1.0 + 0.05 * left + smooth(1e-4), "ux": zero + smooth(1e-4), "uy": zero + smooth(1e-4),
                "T": one + smooth(1e-4)}
    if flow == "rb":  # a layer of convection rolls growing on the hydrostatic state
        _, col = W.rayleigh_benard(3, ny, amp=0.0)
        H, u_c, dT = ny - 1, 0.03, 0.02
        s, kx = torch.sin(math.pi * y / H), 2.0 * math.pi * max(1, round(nx / (2.0 * ny))) / nx
        rho = torch.from_numpy(col["rho"][:, :1].copy()).cuda() * torch.ones_like(x)
        T = torch.from_numpy(col["T"][:, :1].copy()).cuda() * torch.ones_like(x)
        # u = curl of s^2 sin(kx x), zero on both walls
        ux = 0.3 * u_c * 2.0 * s * torch.cos(math.pi * y / H) * torch.sin(kx * x)
        uy = -0.3 * u_c * (kx * H / math.pi) * s * s * torch.cos(kx * x)
        edge = (s > 1e-9).double()
        return {"rho": rho, "ux": ux + edge * smooth(1e-4), "uy": uy + edge * smooth(1e-4),
                "T": T - 0.2 * dT * s * torch.cos(kx * x) + edge * smooth(1e-4)}
    return {"rho": one + smooth(1e-2), "ux": smooth(2e-2), "uy": smooth(2e-2), "T": one + smooth(1e-2)}


def _thermal(case):
    if case["flow"] == "taylor_green":
        return bool(case.get("thermal"))
    return case.get("variant", "corr") != "athermal"


SWEEP_SIZES = ((64, 32), (128, 64), (256, 128), (512, 256), (1024, 512))


def _members(case, seed):
    """The single-lattice cases of a batch or of a burst of requests (sizes as the sweep and the
    request trace have them; the mix is the case's own, not the seed's)."""
    rng = np.random.default_rng(97 + case["count"])
    out = []
    for i in range(case["count"]):
        m = {"kind": "flow", "storage": case["storage"], "rounding": case["rounding"], "seed": int(seed) * 131 + i}
        if case["kind"] == "batch":
            nx, ny = SWEEP_SIZES[int(rng.integers(len(SWEEP_SIZES)))]
            m.update(flow="rb", nx=nx, ny=ny, steps=case["steps"])
        else:
            which, steps = i % 3, int(rng.choice((50, 100, 200)))
            if which == 0:
                m.update(flow="couette", nx=32, ny=128, steps=steps)
            elif which == 1:
                n = int(2 ** rng.integers(7, 11))
                m.update(flow="taylor_green", nx=n, ny=n, thermal=True, steps=steps)
            else:
                nx = int(2 ** rng.integers(7, 12))
                m.update(flow="rb", nx=nx, ny=nx // 2, steps=steps)
        out.append(m)
    return out


def _populations(case, fields):
    """f_bar, h_bar [9][ny][nx] of the fields, as a checkpoint holds them."""
    ref = _Reference(case)
    f, h = ref.initial(fields)
    return torch.stack(f), (torch.stack(h) if ref.thermal else None)


def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "serve":
        s["members"] = []
        for m in _members(case, seed):
            s["members"].append((_problem(m), {k: v.cpu().numpy() for k, v in _fields(m, m["seed"]).items()}, m["steps"]))
        return s
    if case["kind"] == "batch":
        members = _members(case, seed)
        s["lats"] = [tclbm.Lattice(_problem(m)) for m in members]
        s["fields"] = [_fields(m, m["seed"]) for m in members]
        n = [m["nx"] * m["ny"] for m in members]
        s["out"] = {k: torch.empty(sum(n), dtype=torch.float64, device="cuda") for k in FIELDS}
        at = np.concatenate([[0], np.cumsum(n)])
        s["views"] = [{k: s["out"][k][at[i]:at[i + 1]] for k in FIELDS} for i in range(len(n))]
        s["batch"] = tclbm.Batch(s["lats"])
        s["batch"].set_tile(32, 16, False)
        s["batch"].set_tma(128, 32)
        return s
    s["fields"] = _fields(case, seed)
    s["lat"] = tclbm.Lattice(_problem(case))
    n = (case["ny"], case["nx"])
    if case["kind"] == "restart":
        s["f"], s["h"] = _populations(case, s["fields"])
        s["f_out"] = torch.empty_like(s["f"])
        s["h_out"] = torch.empty_like(s["f"]) if s["h"] is not None else None
        return s
    if case.get("host"):
        s["fields"] = {k: v.cpu().numpy() for k, v in s["fields"].items()}
    else:
        s["out"] = {k: torch.empty(n, dtype=torch.float64, device="cuda") for k in FIELDS}
    return s


def _at(t):
    return None if t is None else t.data_ptr()


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "serve":
        reqs = [serve.Request(rid=i, case=c, fields=f, steps=n) for i, (c, f, n) in enumerate(s["members"])]
        done = serve.Server(storage=case["storage"], rounding=case["rounding"]).run(reqs, realtime=False)
        done.sort(key=lambda r: r.rid)
        return [[r.result[k] for k in FIELDS] for r in done]
    if kind == "batch":
        for lat, f in zip(s["lats"], s["fields"]):
            lat.init_fields(f)
        s["batch"].step(case["steps"])
        for lat, v in zip(s["lats"], s["views"]):
            lat.moments_device(v)
        return s["out"]
    lat = s["lat"]
    if kind == "restart":
        tclbm.tclbm_set_populations(lat.handle, _at(s["f"]), _at(s["h"]), True)
        lat.snapshot_velocity()
        lat.step(case["steps"])
        sums = lat.diagnostics()
        tclbm.tclbm_get_populations(lat.handle, _at(s["f_out"]), _at(s["h_out"]), True)
        return {"f": s["f_out"], "h": s["h_out"], "sums": sums}
    lat.init_fields(s["fields"])
    lat.step(case["steps"])
    out = {}
    if case.get("sums"):
        out["sums"] = lat.diagnostics()
    if case.get("host"):
        out.update(lat.moments())
    else:
        lat.moments_device(s["out"])
        out.update(s["out"])
    return out


def work(case):
    """Bytes and operations of one pass: every step reads and writes each population once (18 of
    them with the energy distribution, 9 without), fields or populations in and out are FP64."""
    if case["kind"] in ("batch", "serve"):
        total = {"bytes": 0.0, "flops": 0.0}
        for m in _members(case, 0):
            for k, v in work(m).items():
                total[k] += v
        return total
    nodes, planes = float(case["nx"] * case["ny"]), 18 if _thermal(case) else 9
    size = 4 if case.get("storage", "fp32") == "fp32" else 2
    lu = nodes * case["steps"]
    ends = 2 * planes * 8.0 if case["kind"] == "restart" else 2 * 4 * 8.0
    # moments, gradients and the relaxation of one node: about 500 additions and
    # multiplications with the energy distribution, 200 without
    return {"bytes": lu * 2 * planes * size + nodes * ends, "flops": lu * (500.0 if planes == 18 else 200.0)}


# ------------------------------------------------------------------ the method in 64 bits

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
OPP = (0, 3, 4, 1, 2, 7, 8, 5, 6)
WQ = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4
SIDES = {"x-": (1, 0), "x+": (-1, 0), "y-": (0, 1), "y+": (0, -1)}  # inward normals


def _eq3(rho, m00, m10, m01, E, N, Pi, m21, m12, m22):
    """Populations of nine raw moments."""
    a, b = 0.5 * (E + N), 0.5 * (E - N)
    return [rho * (m00 - E + m22), 0.5 * rho * (m10 + a - m12 - m22), 0.5 * rho * (m01 + b - m21 - m22),
            0.5 * rho * (-m10 + a + m12 - m22), 0.5 * rho * (-m01 + b + m21 - m22),
            0.25 * rho * (Pi + m21 + m12 + m22), 0.25 * rho * (-Pi + m21 - m12 + m22),
            0.25 * rho * (Pi - m21 - m12 + m22), 0.25 * rho * (-Pi - m21 + m12 + m22)]


def _feq(rho, ux, uy, RT):
    X = (1.0 - RT - ux * ux, 0.5 * (RT + ux * ux + ux), 0.5 * (RT + ux * ux - ux))  # e = 0, +1, -1
    Y = (1.0 - RT - uy * uy, 0.5 * (RT + uy * uy + uy), 0.5 * (RT + uy * uy - uy))
    return [rho * X[EX[q]] * Y[EY[q]] for q in range(9)]  # index -1 is the last entry


def _source(rho, ux, uy, ax, ay):
    s = ax * uy + ay * ux
    return _eq3(rho, 0.0, ax, ay, 2.0 * (ax * ux + ay * uy), 2.0 * (ax * ux - ay * uy), s,
                ay * ux * ux + 2.0 * ax * ux * uy, ax * uy * uy + 2.0 * ay * ux * uy, 2.0 * ux * uy * s)


class _Reference:
    """The time step as the paper writes it, on whole arrays in FP64: f, h are lists of nine
    tensors [ny][nx] of the streamed populations with the wall schemes applied."""

    def __init__(self, case):
        d = _problem(case)
        self.d, self.nx, self.ny = d, d["nx"], d["ny"]
        self.thermal, self.corr = bool(d["thermal"]), bool(d["correction"])
        self.b = 2.0 / (d["gamma"] - 1.0)
        self.work = bool(d.get("work")) and self.thermal
        self.walls = [(s, d["walls"][s]) for s in SIDES if d["walls"][s]["kind"] != "periodic"]
        self.xper, self.yper = d["walls"]["x-"]["kind"] == "periodic", d["walls"]["y-"]["kind"] == "periodic"
        o = dict(dtype=torch.float64, device="cuda")
        kx = 2.0 * math.pi / self.nx * torch.arange(self.nx, **o)[None, :]
        ky = 2.0 * math.pi / self.ny * torch.arange(self.ny, **o)[:, None]
        fc = d["force"]
        self.tg = None
        if fc["kind"] == "taylor_green":
            self.tg = (fc["amp"] * torch.sin(kx) * torch.sin(ky), fc["amp"] * torch.cos(kx) * torch.cos(ky))
        self.acc = (fc["ax"], fc["ay"]) if fc["kind"] == "accel" else None
        self.w1_fixed = 1.0 / (d["visc"] / (d["R"] * d["T0"]) + 0.5) if d["w_equal"] else None
        if d["visc_law"] == "w1":
            self.w1_fixed = d["visc"]

    def force(self, rho, at):
        if self.acc:
            return rho * self.acc[0], rho * self.acc[1]
        if self.tg:
            return self.tg[0][at], self.tg[1][at]
        return 0.0, 0.0

    def heq(self, rho, ux, uy, RT):
        uu = ux * ux + uy * uy
        E = 0.5 * (self.b * RT + uu)
        A, B = E + RT, E + 2.0 * RT
        o = [rho * (E - B * uu - 2.0 * RT * A)]
        for q in range(1, 5):
            eu, e2 = EX[q] * ux + EY[q] * uy, EX[q] ** 2 * ux * ux + EY[q] ** 2 * uy * uy
            o.append(0.5 * rho * (A * eu + B * e2 + RT * A))
        return o + [0.25 * rho * B * (EX[q] * EY[q]) * ux * uy for q in range(5, 9)]

    def macro(self, f, h, at=(slice(None), slice(None))):
        rho = sum(f)
        jx = (f[1] - f[3]) + (f[5] - f[6]) + (f[8] - f[7])
        jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8])
        Fx, Fy = self.force(rho, at)
        ux, uy = (jx + 0.5 * Fx) / rho, (jy + 0.5 * Fy) / rho
        if self.thermal:
            sh = sum(h)
            if self.work:
                sh = sh + 0.5 * (Fx * ux + Fy * uy)
            T = 2.0 / (self.b * self.d["R"]) * (sh / rho - 0.5 * (ux * ux + uy * uy))
        else:
            T = torch.full_like(rho, self.d["T0"])
        return rho, ux, uy, T, Fx, Fy

    def initial(self, fields):
        rho, ux, uy = fields["rho"], fields["ux"], fields["uy"]
        T = fields["T"] if self.thermal else torch.full_like(rho, self.d["T0"])
        Fx, Fy = self.force(rho, (slice(None), slice(None)))
        S = _source(rho, ux, uy, Fx / rho, Fy / rho)
        f = [a - 0.5 * s for a, s in zip(_feq(rho, ux, uy, self.d["R"] * T), S)]
        h = None
        if self.thermal:
            h = self.heq(rho, ux, uy, self.d["R"] * T)
            if self.work:
                h = [a - 0.5 * w * (Fx * ux + Fy * uy) for a, w in zip(h, WQ)]
        self.rebuild(f, h)
        return f, h

    def rebuild(self, f, h):
        """The wall schemes on the wall row or column (in place)."""
        R = self.d["R"]
        for side, w in self.walls:
            nxv, nyv = SIDES[side]
            edge = 0 if nxv + nyv > 0 else -1
            near = 1 if edge == 0 else -2

            def line(i):
                return (slice(None), i) if nxv else (i, slice(None))

            b, n = line(edge), line(near)
            span = (slice(None), slice(edge, edge + 1 or None)) if nxv else (slice(edge, edge + 1 or None), slice(None))
            spin = (slice(None), slice(near, near + 1)) if nxv else (slice(near, near + 1), slice(None))
            fb, ff = [a[span].clone() for a in f], [a[spin].clone() for a in f]
            hf = [a[spin].clone() for a in h] if self.thermal else None
            rf, uf, vf, Tf, Ffx, Ffy = self.macro(ff, hf, spin)
            Tw = self.d["T0"]
            if self.thermal:
                Tw = Tf if w["therm"] == "adiabatic" else w["T"]
            one = torch.ones_like(rf)
            if w["kind"] == "zouhe":
                txv, tyv = (0, 1) if nxv else (1, 0)
                en = [EX[q] * nxv + EY[q] * nyv for q in range(9)]
                known = sum(fb[q] for q in range(9) if en[q] == 0) + 2.0 * sum(fb[q] for q in range(9) if en[q] < 0)
                if self.tg:
                    Fx, Fy = self.force(None, span)
                    rw = known - 0.5 * (Fx * nxv + Fy * nyv)
                    an, at = (Fx * nxv + Fy * nyv) / rw, (Fx * txv + Fy * tyv) / rw
                else:
                    ax, ay = self.acc or (0.0, 0.0)
                    an, at = ax * nxv + ay * nyv, ax * txv + ay * tyv
                    rw = known / (1.0 + 0.5 * an)
                ut = w["ux"] * txv + w["uy"] * tyv
                dirs = {(EX[q], EY[q]): q for q in range(9)}
                i_n, i_t, i_m = dirs[nxv, nyv], dirs[txv, tyv], dirs[-txv, -tyv]
                i_p, i_q = dirs[nxv + txv, nyv + tyv], dirs[nxv - txv, nyv - tyv]
                dn = -0.5 * rw * an * (1.0 - ut * ut)
                td = 0.5 * (fb[i_t] - fb[i_m])
                new_n = fb[OPP[i_n]] + dn
                new_p = fb[OPP[i_p]] - td + 0.5 * rw * ut - 0.25 * rw * at - 0.25 * rw * an - 0.5 * dn
                new_q = fb[OPP[i_q]] + td - 0.5 * rw * ut + 0.25 * rw * at - 0.25 * rw * an - 0.5 * dn
                fb[i_n], fb[i_p], fb[i_q] = new_n, new_p, new_q
            elif w["kind"] == "nee":
                e_w, e_f = _feq(rf, w["ux"] * one, w["uy"] * one, R * Tw), _feq(rf, uf, vf, R * Tf)
                fb = [a + (c - e) for a, c, e in zip(e_w, ff, e_f)]
            else:
                rw = w["rho"] * one
                Fx, Fy = self.force(rw, span)
                S = _source(rw, w["ux"], w["uy"], Fx / rw, Fy / rw)
                Te = w["T"] if self.thermal else self.d["T0"]
                fb = [a - 0.5 * s for a, s in zip(_feq(rw, w["ux"] * one, w["uy"] * one, R * Te), S)]
            for q in range(9):
                f[q][span] = fb[q]
            if not self.thermal:
                continue
            if w["kind"] == "equilibrium":
                hb = self.heq(rw, w["ux"] * one, w["uy"] * one, R * w["T"])
                if self.work:
                    hb = [a - 0.5 * g * (Fx * w["ux"] + Fy * w["uy"]) for a, g in zip(hb, WQ)]
            else:
                rb, ub, vb, _, Fbx, Fby = self.macro(fb, hf, span)
                e_w, e_f = self.heq(rb, ub, vb, R * Tw), self.heq(rf, uf, vf, R * Tf)
                if self.work:
                    qb, qf = Fbx * ub + Fby * vb, Ffx * uf + Ffy * vf
                    e_w = [a - 0.5 * g * qb for a, g in zip(e_w, WQ)]
                    e_f = [a - 0.5 * g * qf for a, g in zip(e_f, WQ)]
                hb = [a + (c - e) for a, c, e in zip(e_w, hf, e_f)]
            for q in range(9):
                h[q][span] = hb[q]

    def slope(self, phi, dim, periodic):
        d = 0.5 * (phi.roll(-1, dim) - phi.roll(1, dim))
        if not periodic:
            p, o = (phi.T, d.T) if dim == 1 else (phi, d)
            o[0] = 0.5 * (-3.0 * p[0] + 4.0 * p[1] - p[2])
            o[-1] = 0.5 * (3.0 * p[-1] - 4.0 * p[-2] + p[-3])
        return d

    def step(self, f, h):
        d, R = self.d, self.d["R"]
        rho, ux, uy, T, Fx, Fy = self.macro(f, h)
        RT, ax, ay = R * T, Fx / rho, Fy / rho
        dx = dy = 0.0
        if self.corr:
            dx = self.slope(ux * (1.0 - 3.0 * RT), 1, self.xper)
            dy = self.slope(uy * (1.0 - 3.0 * RT), 0, self.yper)
        if self.w1_fixed is not None:
            w1 = self.w1_fixed
        else:
            mu_p = {"nu": lambda: d["visc"] / RT, "mu": lambda: d["visc"] / (rho * RT),
                    "mu_T": lambda: d["visc"] * (T / d["T0"]) / (rho * RT)}[d["visc_law"]]()
            w1 = 1.0 / (mu_p + 0.5)
        w2, w3, w4 = (w1,) * 3 if d["w_equal"] else (d["w2"], d["w3"], d["w4"])
        ux2, uy2, uxy = ux * ux, uy * uy, ux * uy
        uu = ux2 + uy2
        # raw moments, then central moments about u
        a57, a68 = f[5] + f[7], f[6] + f[8]
        r20, r02 = (f[1] + f[3] + a57 + a68) / rho, (f[2] + f[4] + a57 + a68) / rho
        r11, r22 = (a57 - a68) / rho, (a57 + a68) / rho
        r21, r12 = (f[5] + f[6] - f[7] - f[8]) / rho, (f[5] - f[6] - f[7] + f[8]) / rho
        r10, r01 = ux - 0.5 * ax, uy - 0.5 * ay
        k20, k02 = r20 - 2.0 * ux * r10 + ux2, r02 - 2.0 * uy * r01 + uy2
        k11 = r11 - ux * r01 - uy * r10 + uxy
        k21 = r21 - 2.0 * ux * r11 - uy * r20 + ux2 * r01 + 2.0 * uxy * r10 - ux2 * uy
        k12 = r12 - 2.0 * uy * r11 - ux * r02 + uy2 * r10 + 2.0 * uxy * r01 - uy2 * ux
        k22 = (r22 - 2.0 * uy * r21 - 2.0 * ux * r12 + uy2 * r20 + ux2 * r02 + 4.0 * uxy * r11
               - 2.0 * uxy * (uy * r10 + ux * r01) + ux2 * uy2)
        # relaxation, and back to raw moments
        Pis, Ns = (1.0 - w1) * k11, w1 * 0.5 * (dy - dx) + (1.0 - w1) * (k20 - k02)
        Es = w2 * (2.0 * RT - 0.5 * (dx + dy)) + (1.0 - w2) * (k20 + k02)
        c21, c12, c22 = (1.0 - w3) * k21, (1.0 - w3) * k12, w4 * RT * RT + (1.0 - w4) * k22
        Pi = Pis + uxy - 0.5 * (ax * uy + ay * ux)
        N = Ns + ux2 - uy2 - (ax * ux - ay * uy)
        E = Es + uu - (ax * ux + ay * uy)
        M21 = c21 + 2.0 * ux * Pi + 0.5 * uy * (E + N) - 2.0 * ux2 * uy + 0.5 * ay * ux2 + ax * uxy
        M12 = c12 + 2.0 * uy * Pi + 0.5 * ux * (E - N) - 2.0 * uy2 * ux + 0.5 * ax * uy2 + ay * uxy
        M22 = (c22 + 2.0 * ux * M12 + 2.0 * uy * M21 - 0.5 * uu * E + 0.5 * (ux2 - uy2) * N - 4.0 * uxy * Pi
               + 3.0 * ux2 * uy2 - uxy * (ax * uy + ay * ux))
        S = _source(rho, ux, uy, ax, ay)
        C = _eq3(rho, 0.0, 0.0, 0.0, dx + dy, dx - dy, 0.0, uy * dx, ux * dy, 0.0)
        fo = [a + s + c for a, s, c in zip(_eq3(rho, 1.0, ux - 0.5 * ax, uy - 0.5 * ay, E, N, Pi, M21, M12, M22), S, C)]
        ho = None
        if self.thermal:
            wh = 1.0 / ((1.0 / w1 - 0.5) / d["Pr"] + 0.5)
            feq, heq = _feq(rho, ux, uy, RT), self.heq(rho, ux, uy, RT)
            qw = Fx * ux + Fy * uy if self.work else 0.0
            ho = []
            for q in range(9):
                Z = EX[q] * ux + EY[q] * uy - 0.5 * uu
                K = Z * (d["Pr"] - 1.0) * w1 * (f[q] - feq[q] + 0.5 * S[q] + 0.5 * C[q])
                ho.append(h[q] - wh * (h[q] - heq[q]) + (1.0 - 0.5 * wh) * (K + WQ[q] * qw))
        f = [a.roll((EY[q], EX[q]), (0, 1)) for q, a in enumerate(fo)]
        h = [a.roll((EY[q], EX[q]), (0, 1)) for q, a in enumerate(ho)] if self.thermal else None
        self.rebuild(f, h)
        return f, h

    def sums(self, f, h, before):
        rho, ux, uy, T, _, _ = self.macro(f, h)
        uu = ux * ux + uy * uy
        sh = sum(a.sum() for a in h) if self.thermal else rho.sum() * 0.0
        res = ((ux - before[0]) ** 2 + (uy - before[1]) ** 2).sum() if before else rho.sum() * 0.0
        T_ref = self.d.get("T_ref", self.d["T0"])
        v = [rho.sum(), (rho * ux).sum(), (rho * uy).sum(), sh, (0.5 * rho * uu).sum(), (uy * (T - T_ref)).sum(), res,
             uu.sum()]
        return torch.stack(v).cpu().numpy()


def _exact_flow(case, seed):
    ref = _Reference(case)
    fields = _fields(case, seed)
    f, h = ref.initial(fields)
    before = ref.macro(f, h)[1:3] if case["kind"] == "restart" else None
    for _ in range(case["steps"]):
        f, h = ref.step(f, h)
    out = {}
    if case.get("sums") or case["kind"] == "restart":
        out["sums"] = ref.sums(f, h, before)
    if case["kind"] == "restart":
        out.update(f=torch.stack(f), h=torch.stack(h) if ref.thermal else None)
        return out
    m = ref.macro(f, h)
    out.update({k: m[i].cpu().numpy() if case.get("host") else m[i] for i, k in enumerate(FIELDS)})
    return out


def exact(case, seed):
    if case["kind"] == "flow" or case["kind"] == "restart":
        return _exact_flow(case, seed)
    got = [_exact_flow(dict(m, host=case["kind"] == "serve"), m["seed"]) for m in _members(case, seed)]
    if case["kind"] == "serve":
        return [[g[k] for k in FIELDS] for g in got]
    return {k: torch.cat([g[k].reshape(-1) for g in got]) for k in FIELDS}
