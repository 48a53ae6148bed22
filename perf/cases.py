"""The measured cases of the lattice Boltzmann library: what a user has it do, through its public
entry points (Lattice, Batch, Server, capi), over the range of sizes, velocity sets, storage types and
options that the repository's configurations, tests and benchmark use.

Five kinds of pass:

* "advance":  a lattice that exists already is advanced by a number of levels and its moments and its
              records of those levels are read (a long run, monitored in stretches);
* "solve":    the standing shear wave from its initial state: init, all levels, records and moments;
* "exchange": host fields in, every level's record read on the host while the next level runs, u_y out;
* "batch":    many uneven shear waves in one persistent launch, with their histories;
* "serve":    requests through the request loop until every one has finished, with their histories;
* "dvm":      the reduced discrete velocity method, one run for several collision times.

Results of FP64 lattices and of the DVM are returned in FP64, those of FP32 and 16-bit lattices in FP32,
the type of their arithmetic.  exact() is the same scheme written out in torch in 64 bits.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

from paper_0908_4520_gb300 import Batch, Lattice, capi
from paper_0908_4520_gb300.serve import Server

GH = {"D2Q16-GH": 4, "D2Q36-GH": 6, "D2Q64-GH": 8}
# on-lattice sets: one representative of each fully symmetric shell, a start value for c, the even
# moments <x^2i y^2j> their weights meet (as many as there are unknowns: the weights and c)
SHELLS = {
    "D2Q9": ([(0, 0), (1, 0), (1, 1)], 1.7320508, [(0, 0), (1, 0), (1, 1), (2, 0)]),
    "D2Q17": ([(0, 0), (1, 0), (1, 1), (2, 2), (3, 0)], 1.6434306,
              [(0, 0), (1, 0), (2, 0), (1, 1), (3, 0), (2, 1)]),
    "D2Q37": ([(0, 0), (1, 0), (1, 1), (2, 0), (2, 1), (2, 2), (3, 0), (3, 1)], 1.196979770,
              [(0, 0), (1, 0), (2, 0), (1, 1), (3, 0), (2, 1), (4, 0), (3, 1), (2, 2)]),
}
NQ = {"D2Q16-GH": 16, "D2Q36-GH": 36, "D2Q64-GH": 64, "D2Q9": 9, "D2Q17": 17, "D2Q37": 37}
BYTES = {"f32": 4, "f64": 8, "f16": 2, "bf16": 2}

_BASE = dict(n_eq=3, precision="f32", kn=0.1, kn_convention="lambda", isothermal=False, scheme="second_order",
             streaming="lax_wendroff", force_amp=0.0, force_freq=0.0, u=1e-3)


def _lattice(kind, quadrature, nx, ny, levels, **more):
    return dict(_BASE, kind=kind, quadrature=quadrature, nx=nx, ny=ny, levels=levels, **more)


def listed():
    return [
        # the correctness configuration: one small shear wave in FP64, every level recorded; each level
        # is a few thousand operations, so launches and latency are all there is
        dict(_lattice("solve", "D2Q16-GH", 64, 1, 2000, n_eq=2, precision="f64"), name="small-f64"),
        # one point of the driven-wave sweep (the paper's experiment): FP64, body force, isothermal
        dict(_lattice("solve", "D2Q64-GH", 128, 1, 1500, n_eq=4, precision="f64", isothermal=True,
                      kn_convention="paper", force_amp=1e-4, force_freq=1.0, u=0.0), name="driven-f64"),
        # the grid on which the lattice is compared with the discrete velocity method
        dict(_lattice("solve", "D2Q36-GH", 256, 256, 400), name="subgrid-256"),
        # the plain method at scale, off-lattice set: the headline workload
        dict(_lattice("advance", "D2Q36-GH", 4096, 4096, 32), name="scale-d2q36"),
        # the same with the on-lattice set of degree 9 (exact shift)
        dict(_lattice("advance", "D2Q37", 4096, 4096, 32), name="scale-d2q37"),
        # the precision configuration: fourth order, 16-bit deviations, and its FP32 run
        dict(_lattice("advance", "D2Q64-GH", 2048, 2048, 32, n_eq=4, precision="f16", u=1e-4), name="precision-f16"),
        dict(_lattice("advance", "D2Q64-GH", 2048, 2048, 32, n_eq=4, u=1e-4), name="precision-f32"),
        # a grid that is no multiple of any tile, the smallest product set, second order
        dict(_lattice("advance", "D2Q16-GH", 2502, 1251, 64, n_eq=2), name="ragged-d2q16"),
        # end to end: host fields in, every level's record read while the next one runs, u_y out
        dict(_lattice("exchange", "D2Q36-GH", 1024, 1024, 100), name="exchange-1024"),
        # the batching configuration: 512 uneven instances, FP32
        dict(kind="batch", count=512, mix=9084521, max_steps=800, precision="f32", u=1e-3, name="batch-512"),
        # the serving configuration: mixed small requests and 1024 x 1024 ones, FP16 deviations
        dict(kind="serve", count=60, large=4, mix=9084522, max_steps=400, precision="f16", u=1e-4, name="serve-64"),
        # the discrete velocity method at the driven sweep's seven Knudsen numbers, 20-point rule
        dict(kind="dvm", nodes=20, nx=128, steps=1000, count=7, force_amp=1e-4, force_freq=1.0, u=0.0,
             name="dvm-driven"),
    ]


def _logu(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng: random.Random):
    kind = rng.choice(["advance", "advance", "advance", "solve", "solve", "exchange", "batch", "serve", "dvm"])
    if kind == "batch":
        return dict(kind=kind, count=int(_logu(rng, 24, 512)), mix=rng.randrange(1 << 30),
                    max_steps=int(_logu(rng, 150, 800)), precision=rng.choice(["f32", "f32", "f16", "bf16"]), u=1e-3)
    if kind == "serve":
        return dict(kind=kind, count=int(_logu(rng, 8, 60)), large=rng.randrange(0, 5), mix=rng.randrange(1 << 30),
                    max_steps=int(_logu(rng, 150, 400)), precision=rng.choice(["f16", "f32"]), u=1e-4)
    if kind == "dvm":
        forced = rng.random() < 0.6
        return dict(kind=kind, nodes=rng.choice([4, 6, 8, 20]), nx=int(_logu(rng, 30, 256)),
                    steps=int(_logu(rng, 200, 1000)), count=rng.randrange(1, 9), force_amp=1e-4 if forced else 0.0,
                    force_freq=rng.choice([0.5, 1.0, 2.0]), u=0.0 if forced else 1e-3)
    quad = rng.choice(["D2Q36-GH", "D2Q36-GH", "D2Q16-GH", "D2Q64-GH", "D2Q37", "D2Q9", "D2Q17"])
    product = quad in GH
    n_eq = rng.choice({"D2Q9": [2, 3], "D2Q17": [2, 3]}.get(quad, [1, 2, 3, 4]))
    if kind == "solve":  # small and middle grids, from the initial state
        nx, ny = 2 * int(_logu(rng, 16, 300)), rng.choice([1, 1, 4, int(_logu(rng, 2, 300))])
        precision = rng.choice(["f32", "f64", "f64"])
        forced = product and rng.random() < 0.3
        kn = 10.0 ** rng.uniform(-1.3, 0.3)
        levels = min(2000, 6e8 / (nx * ny * NQ[quad] * (16 if precision == "f64" else 1)))
        if not forced:  # until little of the wave is left, not until nothing is
            levels = min(levels, nx * math.sqrt(NQ[quad]) / 10 * min(4.0 / kn, 5.0))
        levels = int(max(20, levels))
        return _lattice(kind, quad, nx, ny, levels, **dict(_options(rng, quad, n_eq, precision), kn=kn),
                        **(dict(force_amp=1e-4, force_freq=1.0, u=0.0) if forced else {}))
    precision = rng.choice(["f32", "f32", "f16", "bf16"]) if product else "f32"
    cells = _logu(rng, 1 << 16, (1 << 24) * 36 / max(36, NQ[quad]))
    shape = _logu(rng, 0.25, 4.0)
    nx = max(2, 2 * int(math.sqrt(cells * shape) / 2))
    if rng.random() < 0.5:  # a width that whole 16-byte granules fill
        nx = max(8, nx // 8 * 8)
    ny = max(1, int(cells / nx))
    if kind == "exchange":
        nx, ny = min(nx, 1536), min(ny, 1024)
        precision = "f32"
    levels = int(max(8, min(200, 2e10 / (nx * ny * NQ[quad] * (1 if kind == "advance" else 3)))))
    levels = min(levels, 32) if nx * ny > 1 << 22 else levels
    return _lattice(kind, quad, nx, ny, levels, **_options(rng, quad, n_eq, precision),
                    **(dict(u=1e-4) if precision in ("f16", "bf16") else {}))


def _options(rng, quad, n_eq, precision):
    return dict(n_eq=n_eq, precision=precision, kn=10.0 ** rng.uniform(-1.3, 0.3),
                isothermal=rng.random() < 0.2,
                streaming="upwind2" if quad in GH and precision in ("f32", "f64") and rng.random() < 0.15
                else "lax_wendroff")


# ------------------------------------------------------------------ inputs
def _device():
    return torch.device("cuda")


def _fields(case, seed):
    """rho, u_x, u_y, T on the host: the shear wave and a few long waves of its amplitude in every field."""
    nx, ny, u = case["nx"], case["ny"], case["u"]
    rng = np.random.default_rng(seed)
    x = torch.arange(nx, dtype=torch.float64, device=_device()) * (2 * math.pi / nx)
    y = torch.arange(ny, dtype=torch.float64, device=_device()) * (2 * math.pi / ny)
    out = []
    for k, base in enumerate((1.0, 0.0, 0.0, 1.0)):
        f = torch.full((ny, nx), base, dtype=torch.float64, device=_device())
        if k == 2:
            f += u * rng.uniform(0.8, 1.2) * torch.sin(x)[None, :]
        for mx, my in ((1, 1), (2, 1), (1, 2)):
            a, p, q = u * rng.uniform(0.2, 0.5), rng.uniform(0, 2 * math.pi), rng.uniform(0, 2 * math.pi)
            f += a * torch.cos(my * y + q)[:, None] * torch.cos(mx * x + p)[None, :]
        out.append(f.cpu().numpy())
    return out


def _wave(case, seed):
    rng = np.random.default_rng(seed)
    return case["u"] * float(rng.uniform(0.8, 1.2)), case["u"] * float(rng.uniform(0.8, 1.2))


def _force(case, seed):
    return case["force_amp"] * float(np.random.default_rng(seed + 1).uniform(0.8, 1.2))


def _instances(case, seed):
    """A mix of grids, sets and orders that the case fixes, with Knudsen numbers and amplitudes of the seed."""
    mix, rng = np.random.default_rng(case["mix"]), np.random.default_rng(seed)
    out = []
    for i in range(case["count"] + case.get("large", 0)):
        if i >= case["count"]:
            d = dict(quadrature="D2Q36-GH", n_eq=3, nx=1024, ny=1024)
        else:
            d = dict(quadrature=list(GH)[int(mix.integers(0, 3))], n_eq=int(mix.integers(2, 5)),
                     nx=int(2 ** mix.integers(5, 11)), ny=(1, 4)[int(mix.integers(0, 2))])
        out.append(dict(d, kn=float(10.0 ** rng.uniform(-2.0, 1.0)), u0=case["u"] * float(rng.uniform(0.8, 1.2))))
    return [out[i] for i in mix.permutation(len(out))]


def _taus(case, seed):
    base = np.geomspace(0.01, 1.5, 8)[: case["count"]]
    return base * np.random.default_rng(seed).uniform(0.9, 1.1, len(base))


def prepare(case, seed):
    stream = torch.cuda.Stream()
    s = dict(case=case, stream=stream)
    if case["kind"] == "batch":
        s["instances"] = _instances(case, seed)
        s["batch"] = Batch(precision=case["precision"], stream=stream.cuda_stream)
        return s
    if case["kind"] == "serve":
        s["instances"] = _instances(case, seed)
        s["server"] = Server(precision=case["precision"])
        return s
    if case["kind"] == "dvm":
        s["taus"] = _taus(case, seed)
        s["u"], s["force"] = _wave(case, seed)[0], _force(case, seed)
        return s
    s["lattice"] = Lattice(case["quadrature"], case["n_eq"], case["nx"], case["ny"], case["kn"],
                           precision=case["precision"], kn_convention=case["kn_convention"],
                           isothermal=case["isothermal"], scheme=case["scheme"], streaming=case["streaming"],
                           force_amp=_force(case, seed), force_freq=case["force_freq"], stream=stream.cuda_stream)
    s["wave"] = _wave(case, seed)
    if case["kind"] == "exchange":
        s["fields"] = [torch.from_numpy(f).pin_memory().numpy().reshape(-1) for f in _fields(case, seed)]
        s["uy"] = torch.empty(case["nx"] * case["ny"], dtype=torch.float64).pin_memory().numpy()
    else:
        s["moments"] = torch.empty((5, case["ny"], case["nx"]), dtype=torch.float64, device=_device())
    if case["kind"] == "advance":
        s["lattice"].init_fields(*_fields(case, seed))
    return s


# ------------------------------------------------------------------ one pass
def run(s):
    return {"advance": _run_lattice, "solve": _run_lattice, "exchange": _run_exchange, "batch": _run_batch,
            "serve": _run_serve, "dvm": _run_dvm}[s["case"]["kind"]](s)


MOMENTS = {"rho": 0, "u": slice(1, 3), "T": 3, "sxy": 4}
RECORDS = ("amp", "shear", "hnorm")


def _run_lattice(s):
    case, lat = s["case"], s["lattice"]
    with torch.cuda.stream(s["stream"]):
        if case["kind"] == "solve":
            lat.init_shear_wave(*s["wave"])
        lat.step(case["levels"])
        capi.lb_moments_device(lat.h, *(m.data_ptr() for m in s["moments"]))
        rec = lat.diagnostics(case["levels"] + (1 if case["kind"] == "solve" else 0))
        f64 = case["precision"] == "f64"
        out = {k: s["moments"][i] if f64 else s["moments"][i].float() for k, i in MOMENTS.items()}
        out.update({k: rec[k] if f64 else rec[k].astype(np.float32) for k in RECORDS})
    return out


def _run_exchange(s):
    case, lat = s["case"], s["lattice"]
    capi.lb_init_fields(lat.h, *s["fields"])
    rec = []
    for level in range(case["levels"]):
        lat.step(1)
        r = capi.lb_diagnostics_at(lat.h, level)
        rec.append((r.amp, r.shear, r.hnorm))
    capi.lb_moments(lat.h, None, None, s["uy"])
    rec = np.array(rec, dtype=np.float32)
    return {"uy": s["uy"].astype(np.float32), **{k: rec[:, i] for i, k in enumerate(RECORDS)}}


def _histories(found, case):
    """(A, S) histories of all instances in one array each, zero past an instance's last level."""
    n = case["max_steps"] + 1
    amp, shear = np.zeros((len(found), n), dtype=np.float32), np.zeros((len(found), n), dtype=np.float32)
    for i, (a, b) in enumerate(found):
        amp[i, : len(a)], shear[i, : len(b)] = a, b
    return amp, shear


def _run_batch(s):
    case, b = s["case"], s["batch"]
    slots = [b.add(d["quadrature"], d["n_eq"], d["nx"], d["ny"], d["kn"], d["u0"], max_steps=case["max_steps"],
                   stop_ratio=1e-3) for d in s["instances"]]
    b.run().sync()
    amp, shear = _histories([b.history(k) for k in slots], case)
    for k in slots:
        b.remove(k)
    return {"amp": amp, "shear": shear}


def _run_serve(s):
    case, srv = s["case"], s["server"]
    for i, d in enumerate(s["instances"]):
        srv.submit(i, 0.0, d["quadrature"], d["n_eq"], d["nx"], d["ny"], d["kn"], d["u0"],
                   max_steps=case["max_steps"], stop_ratio=0.0)
    done, now = {}, 0.0
    while len(done) < len(s["instances"]):
        srv.step(now)
        now += 1.0
        done.update({r["id"]: r for r in srv.poll()})
    amp, shear = _histories([srv.history(i, case["max_steps"] + 1) for i in range(len(done))], case)
    return {"amp": amp, "shear": shear,
            "rate": np.array([done[i]["decay_rate"] for i in range(len(done))], dtype=np.float32)}


def _run_dvm(s):
    case = s["case"]
    amp, shear = capi.lb_dvm_run_forced(s["taus"], case["nodes"], case["nx"], s["u"], s["force"], case["force_freq"],
                                        case["steps"], stream=s["stream"].cuda_stream)
    return {"amp": amp, "shear": shear}


# ------------------------------------------------------------------ what a pass cannot do without
def _level(q, n_eq, product):
    """Operations of one cell and level: streaming, moments, equilibrium and relaxation, diagnostics."""
    return q * ((20 if product else 0) + 4 + 2 * (n_eq + 1) + 3 + 5)


ON_CHIP = 160e6  # registers, shared memory and L2 of the card: a smaller state need not leave it between levels


def work(case):
    if case["kind"] == "dvm":
        values = case["nodes"] * case["nx"] * case["count"]
        return dict(bytes=16.0 * case["count"] * (case["steps"] + 1), flops=float(values * case["steps"] * 22))
    if case["kind"] in ("batch", "serve"):
        by, fl, size = 0.0, 0.0, BYTES[case["precision"]]
        for d in _instances(case, 0):
            q, cells = NQ[d["quadrature"]], d["nx"] * d["ny"]
            levels = case["max_steps"] + 1
            by += 16 * levels + (2 * q * size * cells * levels if 2 * q * size * cells > ON_CHIP else 0)
            fl += _level(q, d["n_eq"], True) * cells * levels
        return dict(bytes=by, flops=fl)
    q, cells, levels = NQ[case["quadrature"]], case["nx"] * case["ny"], case["levels"]
    size = BYTES[case["precision"]]
    state = 2.0 * q * size * cells
    moving = state * levels if state > ON_CHIP else (state if case["kind"] == "advance" else 0.0)
    ends = {"advance": 5 * 8, "solve": 5 * 8, "exchange": 5 * 8}[case["kind"]] * cells
    return dict(bytes=moving + ends + 64.0 * levels,
                flops=float(_level(q, case["n_eq"], case["quadrature"] in GH) * cells * levels))


# ------------------------------------------------------------------ the same in 64 bits
def _rule(n):
    x, w = np.polynomial.hermite_e.hermegauss(n)
    return x, w / w.sum()


def _shell(e):
    a, b = e
    return sorted({(s * p, t * r) for p, r in ((a, b), (b, a)) for s in (1, -1) for t in (1, -1)})


def _velocities(quadrature):
    """(xi [q, 2], weights [q], integer vectors [q, 2] or None, c) of a set."""
    if quadrature in GH:
        x, w = _rule(GH[quadrature])
        n = len(x)
        return (np.array([(x[i], x[j]) for i in range(n) for j in range(n)]),
                np.array([w[i] * w[j] for i in range(n) for j in range(n)]), None, 0.0)
    reps, c, moments = SHELLS[quadrature]
    shells = [np.array(_shell(e), dtype=float) for e in reps]

    def conditions(c):
        a = np.array([[np.sum((c * e[:, 0]) ** (2 * i) * (c * e[:, 1]) ** (2 * j)) for e in shells]
                      for i, j in moments])
        b = np.array([math.prod(range(1, 2 * i, 2)) * math.prod(range(1, 2 * j, 2)) for i, j in moments], dtype=float)
        return a, b

    a, b = conditions(c)
    w = np.linalg.lstsq(a, b, rcond=None)[0]
    for _ in range(8):  # Newton's method for the weights and c together
        a, b = conditions(c)
        dc = np.array([2 * (i + j) / c for i, j in moments]) * (a @ w)
        step = np.linalg.solve(np.column_stack([a, dc]), b - a @ w)
        w, c = w + step[:-1], c + step[-1]
    e = np.concatenate(shells)
    return c * e, np.concatenate([np.full(len(s), v) for s, v in zip(shells, w)]), e.astype(int), c


def _tensor(v):
    return torch.as_tensor(np.asarray(v), dtype=torch.float64, device=_device())


class _Scheme:
    """One or more lattices of the same set and width (leading axis), each with its collision time and order."""

    def __init__(self, quadrature, n_eq, nx, tau, *, scheme="second_order", streaming="lax_wendroff", isothermal=False,
                 force=None, freq=0.0, observe=True):
        xi, w, self.e, c = _velocities(quadrature)
        self.q, self.dx = len(w), 2 * math.pi / nx
        self.dt = self.dx / c if self.e is not None else self.dx / np.abs(xi).max()
        self.courant = xi * self.dt / self.dx
        tau, n_eq = np.atleast_1d(tau), np.atleast_1d(n_eq)
        first = scheme == "first_order"
        omega = self.dt / tau if first else self.dt / (tau + 0.5 * self.dt)
        col = lambda v: _tensor(v)[:, None]  # noqa: E731
        self.tau, self.omega, self.hdt = col(tau), col(omega), 0.0 if first else 0.5 * self.dt
        self.sigma = col(np.ones_like(omega) if first else 1 - 0.5 * omega)
        self.second = col((n_eq >= 2).astype(float))
        self.isothermal, self.force, self.freq = isothermal, force, freq
        self.w, self.upwind = _tensor(w), streaming == "upwind2"
        self.winv = 1.0 / self.w
        self.project = _tensor([np.ones(self.q), xi[:, 0], xi[:, 1], (xi ** 2).sum(1), xi[:, 0] * xi[:, 1]])
        he = [np.ones_like(xi), xi, xi ** 2 - 1, xi ** 3 - 3 * xi, xi ** 4 - 6 * xi ** 2 + 3]
        top = int(n_eq.max())
        self.terms = [(i, j) for i in range(top + 1) for j in range(top + 1 - i) if i + j > 0]
        self.top = top
        self.mask = [col((n_eq >= i + j).astype(float)) for i, j in self.terms]
        self.basis = _tensor(np.stack([w * he[i][:, 0] * he[j][:, 1] / math.factorial(i) / math.factorial(j)
                                       for i, j in self.terms], axis=1))  # [q, terms]
        self.sin = self.cos = None

    def grid(self, ny, nx):
        x = torch.arange(nx, dtype=torch.float64, device=_device()) * (2 * math.pi / nx)
        self.shape = (ny, nx)
        self.sin, self.cos = (torch.sin(x).expand(ny, nx).reshape(-1), torch.cos(x).expand(ny, nx).reshape(-1))

    # deviations d = f - w, [lattice, q, cells]; moments as (rho - 1, rho u, u, T - 1), [lattice, cells]
    def equilibrium(self, drho, ux, uy, th, force=None):
        one = torch.ones_like(ux)
        cx, cy = [one, ux], [one, uy]
        for k in range(1, self.top):
            cx.append(ux * cx[k] + k * th * cx[k - 1])
            cy.append(uy * cy[k] + k * th * cy[k - 1])
        if force is not None:
            for k in range(self.top, 0, -1):
                cy[k] = cy[k] + k * self.tau * force * cy[k - 1]
        m = torch.stack([s * cx[i] * cy[j] for (i, j), s in zip(self.terms, self.mask)], dim=1)
        m *= (1 + drho)[:, None]
        out = torch.matmul(self.basis, m)
        out += self.w[None, :, None] * drho[:, None]
        return out

    def moments(self, d, level):
        p = torch.matmul(self.project, d)
        drho, jx, jy, en, pxy = p.unbind(1)
        rho = 1 + drho
        g = None
        if self.force:
            g = self.force * math.cos(self.freq * level * self.dt) * self.sin[None]
            jy = jy + self.hdt * rho * g
        ux, uy = jx / rho, jy / rho
        e2 = en - 2 * drho - rho * (ux * ux + uy * uy)
        sig = pxy - self.second * rho * ux * uy
        if g is not None:
            e2 = e2 + 2 * self.hdt * rho * g * uy
            sig = sig + self.second * self.hdt * rho * g * ux
        th = torch.zeros_like(e2) if self.isothermal else e2 / (2 * rho)
        return drho, ux, uy, th, self.sigma * sig, g

    def record(self, d, m):
        n = 2.0 / self.sin.numel()
        h = torch.einsum("q,bqc->b", self.winv, d * d)
        return torch.stack([n * (m[2] @ self.sin), n * (m[4] @ self.cos), h], dim=1)

    def _line(self, f, axis, c):
        sh = [1, -1, 1, 1]
        if not self.upwind:
            fm, fp = torch.roll(f, 1, axis), torch.roll(f, -1, axis)
            c = _tensor(c).view(sh)
            out = f * (1 - c * c)
            out.addcmul_(fm, 0.5 * c * (1 + c)).addcmul_(fp, -0.5 * c * (1 - c))
            return out
        out = torch.empty_like(f)
        for s in (1, -1):
            k = torch.as_tensor(np.where(np.sign(c) == s)[0], device=_device())
            f0 = f[:, k]
            f1, f2 = torch.roll(f0, s, axis), torch.roll(f0, 2 * s, axis)
            a = _tensor(np.abs(c[k.cpu().numpy()])).view(sh)
            out[:, k] = f0 - a / 2 * (3 * f0 - 4 * f1 + f2) + a * a / 2 * (f0 - 2 * f1 + f2)
        return out

    def stream(self, d):
        f = d.view(d.shape[0], self.q, *self.shape)
        if self.e is not None:
            f = torch.stack([torch.roll(f[:, a], (int(ey), int(ex)), (1, 2)) for a, (ex, ey) in enumerate(self.e)], 1)
        else:
            f = self._line(self._line(f, 2, self.courant[:, 1]), 3, self.courant[:, 0])
        return f.reshape(d.shape)

    def solve(self, drho, ux, uy, th, levels):
        """Records of levels 0..levels and the moments of the last one."""
        d = self.equilibrium(drho, ux, uy, torch.zeros_like(th) if self.isothermal else th)
        rec = []
        for n in range(levels + 1):
            m = self.moments(d, n)
            rec.append(self.record(d, m))
            if n < levels:
                eq = self.equilibrium(*m[:4], m[5])
                d = torch.lerp(d, eq, self.omega[:, :, None]) if d.numel() < 1 << 26 else d.mul_(
                    1 - self.omega[:, :, None]).add_(eq.mul_(self.omega[:, :, None]))
                del eq
                d = self.stream(d)
        return torch.stack(rec, 1), m


def _exact_lattice(case, seed):
    tau = case["kn"] * (math.sqrt(2 / math.pi) if case["kn_convention"] == "lambda" else 1.0)
    nx, ny = case["nx"], case["ny"]
    s = _Scheme(case["quadrature"], case["n_eq"], nx, tau, scheme=case["scheme"], streaming=case["streaming"],
                isothermal=case["isothermal"], force=_force(case, seed), freq=case["force_freq"])
    s.grid(ny, nx)
    if case["kind"] == "solve":
        u0, u1 = _wave(case, seed)
        y = torch.arange(ny, dtype=torch.float64, device=_device()) * (2 * math.pi / ny)
        uy = ((u0 + u1 * torch.sin(y)[:, None]) * s.sin.view(ny, nx)).reshape(1, -1)
        zero = torch.zeros_like(uy)
        drho, ux, th = zero, zero, zero
    else:
        drho, ux, uy, th = (_tensor(f).reshape(1, -1) for f in _fields(case, seed))
        drho, th = drho - 1, th - 1
    rec, m = s.solve(drho, ux, uy, th, case["levels"])
    rec = rec[0].cpu().numpy()
    if case["kind"] == "exchange":
        return {"uy": m[2][0].cpu().numpy(), **{k: rec[:-1, i] for i, k in enumerate(RECORDS)}}
    if case["kind"] == "advance":
        rec = rec[1:]
    fields = torch.stack([1 + m[0], m[1], m[2], 1 + m[3], m[4]]).view(5, ny, nx)
    return {**{k: fields[i] for k, i in MOMENTS.items()}, **{k: rec[:, i] for i, k in enumerate(RECORDS)}}


def _exact_instances(case, seed):
    """Shear waves do not depend on y: one row each, instances of one set and width together."""
    ins, n = _instances(case, seed), case["max_steps"] + 1
    amp, shear = np.zeros((len(ins), n)), np.zeros((len(ins), n))
    for quad, nx in sorted({(d["quadrature"], d["nx"]) for d in ins}):
        at = [i for i, d in enumerate(ins) if (d["quadrature"], d["nx"]) == (quad, nx)]
        s = _Scheme(quad, [ins[i]["n_eq"] for i in at], nx, [ins[i]["kn"] * math.sqrt(2 / math.pi) for i in at])
        s.grid(1, nx)
        uy = _tensor([ins[i]["u0"] for i in at])[:, None] * s.sin[None]
        zero = torch.zeros_like(uy)
        rec = s.solve(zero, zero, uy, zero, n - 1)[0].cpu().numpy()
        if case["kind"] == "batch":  # the stop rule sqrt(H / H0) <= 1e-3
            for k in range(len(at)):
                stop = np.flatnonzero(rec[k, 1:, 2] <= 1e-6 * rec[k, 0, 2])
                if len(stop):
                    rec[k, stop[0] + 2:] = 0.0
        amp[at], shear[at] = rec[:, :, 0], rec[:, :, 1]
    return {"amp": amp, "shear": shear, **({"rate": None} if case["kind"] == "serve" else {})}


def _exact_dvm(case, seed):
    xi, w = _rule(case["nodes"])
    nx, steps, tau = case["nx"], case["steps"], _tensor(_taus(case, seed))[:, None, None]
    u0, amp_f, freq = _wave(case, seed)[0], _force(case, seed), case["force_freq"]
    dx = 2 * math.pi / nx
    dt = 0.5 * dx / np.abs(xi).max()
    x = torch.arange(nx, dtype=torch.float64, device=_device()) * dx
    sin, cos, w, wx = torch.sin(x), torch.cos(x), _tensor(w), _tensor(w * xi)
    c, decay = _tensor(xi * dt / dx)[None, :, None], torch.exp(-0.5 * dt / tau)
    g = u0 * sin.expand(len(tau), len(xi), nx)
    gain = lambda a, b: amp_f * (math.sin(freq * b) - math.sin(freq * a)) / freq  # noqa: E731

    def relax(g, a, b):
        u = torch.einsum("k,bkx->bx", w, g)[:, None]
        return u + gain(a, b) * sin + (g - u) * decay

    amp, shear = [], []
    for n in range(steps + 1):
        amp.append(2 / nx * (torch.einsum("k,bkx->bx", w, g) @ sin))
        shear.append(2 / nx * (torch.einsum("k,bkx->bx", wx, g) @ cos))
        if n < steps:
            g = relax(g, n * dt, (n + 0.5) * dt)
            fm, fp = torch.roll(g, 1, 2), torch.roll(g, -1, 2)
            g = g - 0.5 * c * (fp - fm) + 0.5 * c * c * (fp - 2 * g + fm)
            g = relax(g, (n + 0.5) * dt, (n + 1) * dt)
    return {"amp": torch.stack(amp, 1), "shear": torch.stack(shear, 1)}


def exact(case, seed):
    if case["kind"] == "dvm":
        return _exact_dvm(case, seed)
    if case["kind"] in ("batch", "serve"):
        return _exact_instances(case, seed)
    return _exact_lattice(case, seed)
