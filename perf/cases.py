"""The measured workloads: what users of this framework have it do, through lbm.Lattice, lbm.Batch
and lbm.wall_nusselt_objective.

A case is one of five kinds:
  run      a box advanced `steps` steps, then its fields read and, in FP64, the wall Nusselt
           profile, in FP32 its mean (a wall derivative over L nodes lifts the FP32 rounding of single
           nodes by L; in FP16 storage it is noise in a single snapshot and is not read)
  series   a box advanced in short pieces with the hot wall's Nusselt number logged after each
  batch    an ensemble of uneven cavities advanced together, then every member's Nusselt number
  adjoint  J and dJ/dT_w of the wall-Nusselt objective, forward and backward through torch
  read     what a monitor or a checkpoint takes from a state: fields, populations, wall profile
Results are returned at the precision of the populations they come from (FP64, FP32 or FP16
storage); `read` and `adjoint` return them as the framework gives them.
"""
import math

import numpy as np
import torch

from paper_2504_09041_gb300 import lbm

MA = 0.1
BYTES = {"fp64": 8, "fp32": 4, "fp16s": 2}
OUT = {"fp64": torch.float64, "fp32": torch.float32, "fp16s": torch.float16}
# floating-point operations of one node update (multiply-add as two) and links of both lattices
FLOPS = {2: 413.0, 3: 1150.0}
LINKS = {2: 18, 3: 42}
MEMBER_SIDES = (64, 96, 128, 192, 256, 384, 512)


def _run(name, nx, ny, nz, walls, precision, Ra, steps, option="A", Pr=0.71, bulk=1.0):
    case = {"kind": "run", "nx": nx, "ny": ny, "nz": nz, "walls": walls, "precision": precision,
            "Ra": Ra, "Pr": Pr, "steps": steps, "option": option, "bulk": bulk}
    return dict(case, name=name) if name else case


def listed():
    return [
        # the paper's smallest cavity at full precision, advanced toward its steady Nusselt number
        _run("cavity_64_fp64", 64, 64, 1, "cavity", "fp64", 1e4, 500),
        # the time series of a small run: short pieces, one Nusselt number after each
        {"name": "series_96_fp32", "kind": "series", "nx": 96, "ny": 96, "nz": 1, "walls": "cavity",
         "precision": "fp32", "Ra": 1e5, "Pr": 0.71, "steps": 20, "pieces": 8, "option": "A", "bulk": 1.0},
        # Rayleigh-Benard convection in the three storage forms
        _run("rb_1024x512_fp64", 1024, 512, 1, "rb", "fp64", 1e8, 100),
        _run("rb_1024x512_fp32", 1024, 512, 1, "rb", "fp32", 1e8, 400),
        _run("rb_1024x512_fp16s", 1024, 512, 1, "rb", "fp16s", 1e8, 400),
        # the large cubic cavity, FP32 (the headline form) and FP16 storage
        _run("cube_256_fp32", 256, 256, 256, "cavity", "fp32", 1e6, 20),
        _run("cube_256_fp16s", 256, 256, 256, "cavity", "fp16s", 1e6, 20),
        # the cubic cavity at full precision, at the size of the table runs
        _run("cube_128_fp64", 128, 128, 128, "cavity", "fp64", 1e5, 16),
        # a ragged heated layer (periodic x, adiabatic y, hot below) with the option-B attractors
        _run("layer_131x93x77_fp32_b", 131, 93, 77, "layer", "fp32", 1e5, 50, option="B"),
        # the ensemble of 64 uneven cavities
        {"name": "ensemble_64_fp32", "kind": "batch", "count": 64, "precision": "fp32", "steps": 500,
         "largest": 512, "draws": 4},
        # the design gradient: 256-point hot-wall profile, 2000 steps
        {"name": "adjoint_256", "kind": "adjoint", "nx": 256, "ny": 256, "precision": "fp32",
         "Ra": 1e5, "Pr": 0.71, "steps": 2000, "option": "A"},
        # fields, populations and wall profile of a 3D state, as a monitor or a converter reads them
        {"name": "read_160_fp32", "kind": "read", "nx": 160, "ny": 160, "nz": 160, "walls": "cavity",
         "precision": "fp32", "Ra": 1e6, "Pr": 0.71, "steps": 0, "option": "A", "bulk": 1.0},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["run2", "run2", "run3", "run3", "series", "batch", "adjoint", "read"])
    prec = rng.choice(["fp64", "fp32", "fp16s"])
    Ra = 10.0 ** rng.uniform(4, 6)
    Pr = round(rng.uniform(0.71, 7.0), 3)
    option = rng.choice(["A", "A", "A", "B"])
    bulk = rng.choice([1.0, 1.0, 1.0, 1.2])
    if kind == "run2":
        nx, ny = _log_int(rng, 48, 2048), _log_int(rng, 48, 1024)
        walls = rng.choice(["cavity", "rb"])
        steps = max(20, min(500, int((2.0e7 if prec == "fp64" else 1.0e8) / (nx * ny))))
        return _run("", nx, ny, 1, walls, prec, Ra, steps, option, Pr, bulk)
    if kind in ("run3", "read"):
        nx, ny, nz = (_log_int(rng, 24, 224) for _ in range(3))
        walls = rng.choice(["cavity", "layer"])
        c = _run("", nx, ny, nz, walls, prec, Ra,
                 max(4, min(100, int((1.0e7 if prec == "fp64" else 1.0e8) / (nx * ny * nz)))), option, Pr, bulk)
        if kind == "read":
            c.update(kind="read", steps=0, option="A", bulk=1.0)
        return c
    if kind == "series":
        c = _run("", _log_int(rng, 32, 256), _log_int(rng, 32, 256), 1, "cavity",
                 rng.choice(["fp64", "fp32"]), Ra, rng.randint(5, 60), option, Pr, bulk)
        c.update(kind="series", pieces=rng.randint(2, 10))
        return c
    if kind == "batch":
        return {"kind": "batch", "count": _log_int(rng, 4, 64), "precision": "fp32",
                "steps": rng.randint(50, 300), "largest": rng.choice([192, 256, 384, 512]),
                "draws": rng.randint(0, 10**6)}
    return {"kind": "adjoint", "nx": _log_int(rng, 48, 320), "ny": _log_int(rng, 48, 256), "precision": "fp32",
            "Ra": Ra, "Pr": Pr, "steps": rng.randint(100, 900), "option": option}


# --------------------------------------------------------------------------------------------
# Inputs
# --------------------------------------------------------------------------------------------

_E2 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
_E27 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
        (1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1),
        (-1, 0, -1), (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1), (1, 1, 1), (-1, 1, 1),
        (1, -1, 1), (-1, -1, 1), (1, 1, -1), (-1, 1, -1), (1, -1, -1), (-1, -1, -1)]
_E15 = _E27[:7] + _E27[19:]


def _links(dim):
    """Link vectors and rest weights of the flow and the energy lattice."""
    if dim == 2:
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
        return (_E2, w), (_E2, w)
    return ((_E27, [8 / 27] + [2 / 27] * 6 + [1 / 54] * 12 + [1 / 216] * 8),
            (_E15, [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8))


def _dim(case):
    return 2 if case.get("nz", 1) == 1 else 3


def _walls(case):
    dim = _dim(case)
    kind = case.get("walls", "cavity")
    if kind == "cavity":
        return lbm.Walls.cavity(dim)
    if kind == "rb":
        return lbm.Walls.rayleigh_benard(perturb=0.0)
    return lbm.Walls((0, 0, 1, 1, 2, 2), (0, 0, 0, 0, 1.0, 0.0), 0.5, 0.5, 2)


def _start(case, seed):
    """A smooth seeded state: one convection roll in the plane of gravity and a temperature that
    meets the walls, with a few modes on top.  Returns populations (f, g), FP64, on the GPU."""
    dim = _dim(case)
    w = _walls(case)
    shape = (case.get("nz", 1), case["ny"], case["nx"])
    rng = np.random.default_rng(seed)
    up = 1 if dim == 2 else 2
    ext = {0: shape[2], 1: shape[1], 2: shape[0]}
    pos = {}
    for ax in range(3):
        v = [1, 1, 1]
        v[2 - ax] = ext[ax]
        pos[ax] = ((torch.arange(ext[ax], dtype=torch.float64, device="cuda") + 0.5) / ext[ax]).view(v)
    amp = (0.3 + 0.3 * rng.random()) * MA / math.sqrt(3.0) * (1 if rng.random() < 0.5 else -1)
    per = w.face[0] == lbm.LBM_PERIODIC
    ph = 2 * math.pi * rng.random()
    sx = torch.sin(2 * math.pi * pos[0] + ph) if per else torch.sin(math.pi * pos[0]) ** 2
    dx = (2 * math.pi * torch.cos(2 * math.pi * pos[0] + ph) if per else math.pi * torch.sin(2 * math.pi * pos[0])) / ext[0]
    sy, dy = torch.sin(math.pi * pos[up]) ** 2, math.pi * torch.sin(2 * math.pi * pos[up]) / ext[up]
    scale = amp * min(ext[0], ext[up]) / math.pi / 2
    mid = (0.6 + 0.4 * torch.sin(math.pi * pos[1])) if dim == 3 else 1.0
    u = [torch.zeros(shape, dtype=torch.float64, device="cuda") for _ in range(3)]
    u[0] = u[0] + scale * sx * dy * mid
    u[up] = u[up] - scale * dx * sy * mid
    if dim == 3:     # and a weaker roll in the horizontal plane
        b = 0.4 * amp * min(ext[0], ext[1]) / math.pi / 2 * torch.sin(math.pi * pos[2])
        u[0] = u[0] + b * sx * math.pi * torch.sin(2 * math.pi * pos[1]) / ext[1]
        u[1] = u[1] - b * dx * torch.sin(math.pi * pos[1]) ** 2
    hot = next(f for f in range(6) if w.face[f] == lbm.LBM_WALL_FIXED_T)
    ax = hot // 2
    T = w.T_wall[hot] + (w.T_wall[hot + 1] - w.T_wall[hot]) * pos[ax] + torch.zeros(shape, dtype=torch.float64, device="cuda")
    other = up if ax == 0 else 0
    for k in (1, 2, 3):
        a, p = 0.08 * rng.uniform(-1, 1) / k, 2 * math.pi * rng.random()
        T = T + a * torch.sin(k * math.pi * pos[ax]) * torch.cos(2 * math.pi * k * pos[other] + p)
    (ef, wf), (eg, wg) = _links(dim)
    u2 = u[0] ** 2 + u[1] ** 2 + u[2] ** 2
    f = torch.empty((len(wf), *shape), dtype=torch.float64, device="cuda")
    g = torch.empty((len(wg), *shape), dtype=torch.float64, device="cuda")
    for out, es, ws, m in ((f, ef, wf, 1.0), (g, eg, wg, T)):
        for a, (e, wa) in enumerate(zip(es, ws)):
            eu = e[0] * u[0] + e[1] * u[1] + e[2] * u[2]
            out[a] = wa * m * (1 + 3 * eu + 4.5 * eu * eu - 1.5 * u2)
    return f, g


def _profile(seed, n):
    a = np.random.default_rng(seed).uniform(-1.0, 1.0, 4)
    j = np.arange(n) + 0.5
    return 1.0 + 0.05 * sum(a[k] * np.sin(math.pi * (k + 1) * j / n) for k in range(4))


def _ensemble(case):
    rng = np.random.default_rng(case["draws"])
    side = rng.choice(np.asarray([s for s in MEMBER_SIDES if s <= case["largest"]]), size=case["count"])
    Ra = 10.0 ** rng.uniform(3.0, 7.0, case["count"])
    Pr = rng.uniform(0.71, 7.0, case["count"])
    return [(int(s), int(s)) for s in side], Ra.tolist(), Pr.tolist()


def _member_walls(case, seed):
    walls = []
    for k in range(case["count"]):
        w = lbm.Walls.cavity(2)
        w.seed, w.perturb = seed * 1000 + k, 0.05
        walls.append(w)
    return walls


def prepare(case, seed):
    if case["kind"] == "batch":
        sizes, Ra, Pr = _ensemble(case)
        b = lbm.Batch(sizes, Ra, Pr, Ma=MA, walls=_member_walls(case, seed), precision=case["precision"])
        b.tune(20)
        return {"case": case, "batch": b}
    dim = _dim(case)
    lat = lbm.Lattice("d2q9" if dim == 2 else "d3q27", case["nx"], case["ny"], case.get("nz", 1), Ra=case["Ra"],
                      Pr=case["Pr"], Ma=MA, walls=_walls(case), precision=case["precision"])
    if case["option"] == "B":
        lat.set_param("g_attractors", 1)
    if case.get("bulk", 1.0) != 1.0:
        lat.set_param("omega_bulk", case["bulk"])
    lat.set_populations(*_start(case, seed))
    if case["kind"] == "adjoint":
        T_w = torch.tensor(_profile(seed, case["ny"]), device="cuda", requires_grad=True)
        return {"case": case, "lat": lat, "T_w": T_w, "state0": lat.get_state()}
    return {"case": case, "lat": lat}


# --------------------------------------------------------------------------------------------
# One pass
# --------------------------------------------------------------------------------------------

def _hot_face(case):
    return {"cavity": 0, "rb": 2, "layer": 4}[case.get("walls", "cavity")]


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "batch":
        b = state["batch"]
        b.step(case["steps"])
        b.sync()
        nu = [b.nusselt(k, 0)[:3] for k in range(case["count"])]
        f, g = b.get_populations(0)
        return {"nu": np.array(nu, dtype=np.float32), "f0": f, "g0": g}
    lat = state["lat"]
    if kind == "adjoint":
        T_w = state["T_w"]
        T_w.grad = None
        J = lbm.wall_nusselt_objective(lat, state["state0"], case["steps"], 1, 0)(T_w)
        J.backward()
        return {"J": J.detach(), "dJ_dTw": T_w.grad}
    face = _hot_face(case)
    if kind == "series":
        log = []
        for _ in range(case["pieces"]):
            lat.step(case["steps"])
            log += lat.nusselt(face)[:3]
        return {"nu": log, "T": lat.fields()["T"].to(OUT[case["precision"]])}
    if kind == "read":
        f, g = lat.get_populations(device=True)
        return {"fields": lat.fields(), "nu": lat.nusselt_profile(face), "f": f, "g": g}
    lat.step(case["steps"])
    out = OUT[case["precision"]]
    res = {"fields": {k: v.to(out) for k, v in lat.fields().items()}}
    if case["precision"] != "fp16s":
        res["nu"] = lat.nusselt_profile(face) if case["precision"] == "fp64" else lat.nusselt(face)[0]
    return res


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n = sum(a * b for a, b in _ensemble(case)[0])
        return {"bytes": case["steps"] * n * 2.0 * 18 * BYTES[case["precision"]], "flops": case["steps"] * n * FLOPS[2]}
    dim = _dim(case)
    n = float(case["nx"] * case["ny"] * case.get("nz", 1))
    sb = BYTES[case["precision"]]
    q = LINKS[dim]
    if kind == "read":
        # the state read once; five fields and the populations written in FP64
        return {"bytes": n * (q * sb + 5 * 8 + q * 8), "flops": n * 3.0 * q}
    steps = case["steps"] * case.get("pieces", 1)
    if kind == "adjoint":
        # per step: the forward update, and the reverse step that reads the state and the adjoint
        # (8-byte values) and writes the adjoint; the reverse product is at least twice the update
        return {"bytes": steps * n * (2.0 * q * sb + q * sb + 2.0 * q * 8), "flops": steps * n * 3.0 * FLOPS[2]}
    return {"bytes": steps * n * 2.0 * q * sb, "flops": steps * n * FLOPS[dim]}


# --------------------------------------------------------------------------------------------
# The same results in 64 bits: the method written out on torch tensors, moments of full
# populations, no deviation form (arXiv 2504.09041, Sec. 5-6 and App. A-C)
# --------------------------------------------------------------------------------------------

class _Box:
    def __init__(self, case):
        w = _walls(case)
        dim = self.dim = _dim(case)
        self.kind = list(w.face)
        if dim == 2:
            self.kind[4] = self.kind[5] = 0
        self.T_wall = list(w.T_wall)
        self.shape = (case.get("nz", 1), case["ny"], case["nx"])
        nz, ny, nx = self.shape
        n = self.n = nx * ny * nz
        fixed = [f for f in range(6) if self.kind[f] == 2]
        self.L = {0: nx, 1: ny, 2: nz}[fixed[0] // 2]
        self.dT = max(self.T_wall[f] for f in fixed) - min(self.T_wall[f] for f in fixed)
        U = MA / math.sqrt(3.0)
        nu = U * self.L * math.sqrt(case["Pr"] / case["Ra"])
        self.gbeta = U * U / (self.L * self.dT)
        self.up = w.gravity_axis
        self.om_nu = 1 / (3 * nu + 0.5)
        self.om_al = 1 / (3 * nu / case["Pr"] + 0.5)
        self.bulk = case.get("bulk", 1.0)
        self.option = case.get("option", "A")
        (self.ef, self.wf), (self.eg, self.wg) = _links(dim)
        self.idx_f, _ = self._table(self.ef)
        self.idx_g, hit = self._table(self.eg)
        wg = torch.tensor(self.wg, dtype=torch.float64, device="cuda").view(-1, 1, 1, 1)
        self.sign = torch.ones(hit.shape, dtype=torch.float64, device="cuda")
        self.add = torch.zeros(hit.shape, dtype=torch.float64, device="cuda")
        self.design = None
        for f in fixed:
            m = hit == f
            self.sign[m] = -1.0
            if f == 0:
                self.design = 2 * wg * m
            self.add += 2 * wg * m * self.T_wall[f]
        order = [[e[2] + 1, e[1] + 1, e[0] + 1] for e in self.ef]
        self.to_cube = torch.tensor([0] * len(order), device="cuda")
        side = 3 if dim == 3 else 1
        for a, (c, b, x) in enumerate(order):
            at = (c if dim == 3 else 0) * 9 + b * 3 + x
            self.to_cube[at] = a
        self.from_cube = torch.argsort(self.to_cube)
        self.cube = (side, 3, 3)

    def _table(self, es):
        """Flat source index of every link, and the face whose rule a crossing link takes (-1 none):
        the crossed face that comes last in the order -z, -y, -x, +x, +y, +z."""
        nz, ny, nx = self.shape
        lin = torch.arange(self.n, device="cuda").view(self.shape)
        src = torch.stack([torch.roll(lin, (e[2], e[1], e[0]), (0, 1, 2)) + a * self.n for a, e in enumerate(es)])
        hit = torch.full(src.shape, -1, dtype=torch.int8, device="cuda")
        opp = [es.index(tuple(-c for c in e)) for e in es]
        for f in (4, 2, 0, 1, 3, 5):
            if self.kind[f] == 0:
                continue
            ax, hi = f // 2, f % 2
            sl = [slice(None)] * 3
            sl[2 - ax] = slice(-1, None) if hi else slice(0, 1)
            for a, e in enumerate(es):
                if e[ax] == (-1 if hi else 1):
                    src[a][tuple(sl)] = lin[tuple(sl)] + opp[a] * self.n
                    hit[a][tuple(sl)] = f
        return src.view(-1), hit

    def stream(self, f, g, T_w=None):
        f = torch.gather(f.reshape(-1), 0, self.idx_f).view(len(self.wf), *self.shape)
        g = torch.gather(g.reshape(-1), 0, self.idx_g).view(len(self.wg), *self.shape) * self.sign
        if T_w is None:
            return f, g + self.add
        return f, g + (self.add + self.design * (T_w.view(1, 1, -1, 1) - self.T_wall[0]))

    def macro(self, f, g):
        T = g.sum(0)
        F = [None, None, None]
        F[self.up] = self.gbeta * (T - 0.5)
        rho = f.sum(0)
        u = []
        for d in range(self.dim):
            j = sum(f[a] if e[d] > 0 else -f[a] for a, e in enumerate(self.ef) if e[d])
            u.append((j + (0.5 * F[d] if F[d] is not None else 0.0)) / rho)
        return rho, u, T, F

    def central(self, f, u):
        P = f[self.to_cube].view(*self.cube, *self.shape)
        for ax in range(self.dim):
            a, b, c = P.unbind(2 - ax)
            d, s = c - a, c + a
            k0 = s + b
            P = torch.stack((k0, d - u[ax] * k0, s - 2 * u[ax] * d + u[ax] ** 2 * k0), 2 - ax)
        return P

    def uncentral(self, P, u):
        for ax in range(self.dim):
            k0, k1, k2 = P.unbind(2 - ax)
            r1 = k1 + u[ax] * k0
            r2 = k2 + 2 * u[ax] * k1 + u[ax] ** 2 * k0
            P = torch.stack((0.5 * (r2 - r1), k0 - r2, 0.5 * (r2 + r1)), 2 - ax)
        return P.reshape(-1, *self.shape)[self.from_cube]

    def flow2(self, k, rho, F):
        k = k[0]
        on = self.om_nu
        X, Y = (0.0 if v is None else v / rho for v in F[:2])
        Fx, Fy = (0.0 if v is None else v for v in F[:2])
        t10, t01 = 0.5 * Fx, 0.5 * Fy
        tr = (1 - self.bulk) * (k[0][2] + k[2][0]) + self.bulk * 2 / 3 * rho
        de = (1 - on) * (k[0][2] - k[2][0])
        t20, t02, t11 = 0.5 * (tr + de), 0.5 * (tr - de), (1 - on) * k[1][1]
        z = torch.zeros_like(rho)
        t21 = 0.5 * (2 * X * k[1][1] + Y * k[0][2])
        t12 = 0.5 * (X * k[2][0] + 2 * Y * k[1][1])
        t22 = (t20 * t02 + 2 * t11 * t11) / rho + (X * k[2][1] + Y * k[1][2])
        return torch.stack([torch.stack([z + v for v in r]) for r in
                            ((rho, t10, t20), (t01, t11, t21), (t02, t12, t22))])[None]

    def energy2(self, n, T):
        n = n[0]
        oa = self.om_al
        z = torch.zeros_like(T)
        t10, t01 = (1 - oa) * n[0][1], (1 - oa) * n[1][0]
        t20 = t02 = T / 3
        if self.option == "A":
            t21, t12, t22 = 2 / 9 * t01, 2 / 9 * t10, (t20 + t02) / 6
        else:
            t21, t12, t22 = 2 / 3 / T * t20 * t01, 2 / 3 / T * t02 * t10, t20 * t02 / T
        return torch.stack([torch.stack([z + v for v in r]) for r in ((T, t10, t20), (t01, z, t21), (t02, t12, t22))])[None]

    def flow3(self, P, rho, F):
        k = lambda a, b, c: P[c][b][a]  # noqa: E731
        on = self.om_nu
        X, Y, Z = (torch.zeros_like(rho) if v is None else v / rho for v in F)
        t = {(0, 0, 0): rho, (1, 0, 0): 0.5 * X * rho, (0, 1, 0): 0.5 * Y * rho, (0, 0, 1): 0.5 * Z * rho}
        for m in ((1, 1, 0), (1, 0, 1), (0, 1, 1)):
            t[m] = (1 - on) * k(*m)
        tr = (1 - self.bulk) * (k(2, 0, 0) + k(0, 2, 0) + k(0, 0, 2)) + self.bulk * rho
        d1, d2 = (1 - on) * (k(2, 0, 0) - k(0, 2, 0)), (1 - on) * (k(2, 0, 0) - k(0, 0, 2))
        t[2, 0, 0], t[0, 2, 0], t[0, 0, 2] = (tr + d1 + d2) / 3, (tr - 2 * d1 + d2) / 3, (tr + d1 - 2 * d2) / 3

        def source(a, b, c):
            s = 0.0
            for v, m, cnt in ((X, (a - 1, b, c), a), (Y, (a, b - 1, c), b), (Z, (a, b, c - 1), c)):
                if cnt:
                    s = s + cnt * v * k(*m)
            return 0.5 * s

        for m in ((1, 2, 0), (1, 0, 2), (2, 1, 0), (0, 1, 2), (2, 0, 1), (0, 2, 1), (1, 1, 1)):
            t[m] = source(*m)
        i = 1 / rho
        q = lambda a, b, c: t[a, b, c]  # noqa: E731
        t[2, 2, 0] = i * (q(2, 0, 0) * q(0, 2, 0) + 2 * q(1, 1, 0) ** 2) + source(2, 2, 0)
        t[2, 0, 2] = i * (q(2, 0, 0) * q(0, 0, 2) + 2 * q(1, 0, 1) ** 2) + source(2, 0, 2)
        t[0, 2, 2] = i * (q(0, 2, 0) * q(0, 0, 2) + 2 * q(0, 1, 1) ** 2) + source(0, 2, 2)
        t[2, 1, 1] = i * (q(2, 0, 0) * q(0, 1, 1) + 2 * q(1, 1, 0) * q(1, 0, 1)) + source(2, 1, 1)
        t[1, 2, 1] = i * (q(0, 2, 0) * q(1, 0, 1) + 2 * q(1, 1, 0) * q(0, 1, 1)) + source(1, 2, 1)
        t[1, 1, 2] = i * (q(0, 0, 2) * q(1, 1, 0) + 2 * q(0, 1, 1) * q(1, 0, 1)) + source(1, 1, 2)
        t[1, 2, 2] = 0.4 * i * (q(0, 2, 0) * q(1, 0, 2) + q(0, 0, 2) * q(1, 2, 0) + 4 * q(0, 1, 1) * q(1, 1, 1)
                                + 2 * (q(1, 0, 1) * q(0, 2, 1) + q(1, 1, 0) * q(0, 1, 2))) + source(1, 2, 2)
        t[2, 1, 2] = 0.4 * i * (q(2, 0, 0) * q(0, 1, 2) + q(0, 0, 2) * q(2, 1, 0) + 4 * q(1, 0, 1) * q(1, 1, 1)
                                + 2 * (q(1, 1, 0) * q(1, 0, 2) + q(0, 1, 1) * q(2, 0, 1))) + source(2, 1, 2)
        t[2, 2, 1] = 0.4 * i * (q(2, 0, 0) * q(0, 2, 1) + q(0, 2, 0) * q(2, 0, 1) + 4 * q(1, 1, 0) * q(1, 1, 1)
                                + 2 * (q(0, 1, 1) * q(2, 1, 0) + q(1, 0, 1) * q(1, 2, 0))) + source(2, 2, 1)
        t[2, 2, 2] = i / 3 * (q(2, 0, 0) * q(0, 2, 2) + q(0, 2, 0) * q(2, 0, 2) + q(0, 0, 2) * q(2, 2, 0)
                              + 4 * (q(1, 1, 0) * q(1, 1, 2) + q(1, 0, 1) * q(1, 2, 1) + q(0, 1, 1) * q(2, 1, 1))) \
            + source(2, 2, 2)
        out = torch.empty_like(P)
        for (a, b, c), v in t.items():
            out[c][b][a] = v
        return out

    def energy3(self, g, T, u):
        """D3Q15 (App. C): the free energy rates are 1, so of the pre-collision central moments only
        those of order 1 survive; back to populations through the raw moments."""
        oa = self.om_al
        ux, uy, uz = u
        first = [sum(g[b] if e[d] > 0 else -g[b] for b, e in enumerate(self.eg) if e[d]) for d in range(3)]
        t100, t010, t001 = ((1 - oa) * (first[d] - u[d] * T) for d in range(3))
        t2 = T / 3
        if self.option == "A":
            t120, t012, t201, t220 = 2 / 9 * t100, 2 / 9 * t010, 2 / 9 * t001, T / 9
        else:
            t120, t012, t201, t220 = 2 / 3 / T * t2 * t100, 2 / 3 / T * t2 * t010, 2 / 3 / T * t2 * t001, t2 * t2 / T
        q100, q010, q001 = t100 + ux * T, t010 + uy * T, t001 + uz * T
        q200, q020, q002 = t2 + ux * (t100 + q100), t2 + uy * (t010 + q010), t2 + uz * (t001 + q001)
        q110, q101, q011 = ux * t010 + uy * q100, ux * t001 + uz * q100, uy * t001 + uz * q010
        # third order: the shift of each axis in turn
        q120 = t120 + uy * uy * t100 + ux * q020
        q012 = t012 + uz * uz * t010 + uy * q002
        q201 = t201 + ux * ux * t001 + uz * q200
        q111 = ux * uy * t001 + uz * q110
        # order 4: sum g (e_x - ux)^2 (e_y - uy)^2 = t220, with e_x^2 e_y = e_y e_z^2 on these links
        x2y = q012 - ux * (2 * q110 - ux * q010)          # sum g (e_x - ux)^2 e_y
        q220 = t220 + uy * (2 * x2y - uy * t2) + ux * (2 * q120 - ux * q020)
        out = torch.empty_like(g)
        out[0] = T - q200 - q020 - q002 + 2 * q220
        for b, e in enumerate(self.eg):
            if b == 0:
                continue
            x, y, z = e
            if abs(x) + abs(y) + abs(z) == 1:
                two, one, three = ((q200, q100, q120), (q020, q010, q012), (q002, q001, q201))[0 if x else 1 if y else 2]
                out[b] = 0.5 * (two - q220 + (x + y + z) * (one - three))
            else:
                out[b] = 0.125 * (q220 + x * q120 + y * q012 + z * q201 + x * y * q110 + x * z * q101
                                  + y * z * q011 + x * y * z * q111)
        return out

    def step(self, f, g, T_w=None):
        f, g = self.stream(f, g, T_w)
        rho, u, T, F = self.macro(f, g)
        if self.dim == 2:
            return (self.uncentral(self.flow2(self.central(f, u), rho, F), u),
                    self.uncentral(self.energy2(self.central(g, u), T), u))
        f = self.uncentral(self.flow3(self.central(f, u), rho, F), u)
        return f, self.energy3(g, T, u)

    def nusselt(self, g, face, T_w=None):
        _, g = self.stream(torch.zeros((len(self.wf), *self.shape), dtype=g.dtype, device=g.device), g, T_w)
        ax, hi = face // 2, face % 2
        T = g.sum(0).movedim(2 - ax, 0)
        T1, T2 = (T[-1], T[-2]) if hi else (T[0], T[1])
        s = 1.0 if self.T_wall[face] >= 0.5 else -1.0
        return (-s * self.L / self.dT * (-8 / 3 * self.T_wall[face] + 3 * T1 - T2 / 3)).reshape(-1)

    def fields(self, f, g):
        rho, u, T, _ = self.macro(*self.stream(f, g))
        u += [torch.zeros_like(rho)] * (3 - len(u))
        return {"rho": rho, "ux": u[0], "uy": u[1], "uz": u[2], "T": T}


def _exact_adjoint(case, seed):
    box = _Box(case)
    f, g = _start(case, seed)
    n, seg = case["steps"], int(math.isqrt(case["steps"]))
    T_w = torch.tensor(_profile(seed, case["ny"]), device="cuda")
    kept = []
    with torch.no_grad():
        for s in range(n):
            if s % seg == 0:
                kept.append((f, g))
            f, g = box.step(f, g, T_w)
    T_w.requires_grad_(True)
    f.requires_grad_(True)
    g.requires_grad_(True)
    J = box.nusselt(g, 1, T_w).mean()
    back = torch.autograd.grad(J, (f, g, T_w), allow_unused=True)
    lf = torch.zeros_like(f) if back[0] is None else back[0]
    lg = back[1]
    grad = torch.zeros_like(T_w) if back[2] is None else back[2]
    for m in range(len(kept) - 1, -1, -1):
        f0, g0 = (v.detach().requires_grad_(True) for v in kept[m])
        a, b = f0, g0
        for _ in range(min(n, (m + 1) * seg) - m * seg):
            a, b = box.step(a, b, T_w)
        lf, lg, gt = torch.autograd.grad((a, b), (f0, g0, T_w), (lf, lg))
        grad = grad + gt
    return {"J": J.detach(), "dJ_dTw": grad.detach()}


def exact(case, seed):
    kind = case["kind"]
    if kind == "adjoint":
        return _exact_adjoint(case, seed)
    if kind == "batch":
        return None      # starts from the framework's own perturbation; its members are `run` cases
    with torch.no_grad():
        box = _Box(case)
        f, g = _start(case, seed)
        face = _hot_face(case)
        log = []
        for _ in range(case.get("pieces", 1)):
            for _ in range(case["steps"]):
                f, g = box.step(f, g)
            if kind == "series":
                nu = box.nusselt(g, face)
                log += [nu.mean(), nu.max(), nu.min()]
        fields = box.fields(f, g)
        if kind == "series":
            return {"nu": log, "T": fields["T"]}
        nu = box.nusselt(g, face)
        if kind == "read":
            return {"fields": fields, "nu": nu, "f": f, "g": g}
        return {"fields": fields, "nu": {"fp64": nu, "fp32": float(nu.mean()), "fp16s": None}[case["precision"]]}
