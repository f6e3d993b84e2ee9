"""The performance cases of the library: what its users have it do, through its public entry points.

A pass is a piece of work as a program writes it: set the initial state, take the steps, read the
fields (or the history, or the map) back.  Handles, absorbing profiles and initial fields are what
the program holds before the call.  Fields of FP32 and 16-bit lattices are kept in single precision,
those of FP64 lattices in double, as a program stores its snapshots.

The listed cases:

  small_100_f32     the 100^2 pulse of the paper's Sec. 4.1 set-up, 300 steps: the smallest solve, where
                    launches and latency count
  history_200_f32   the decay study of Sec. 4.1: 200^2, Orszag layer, the error norm every 10 steps
  flow_1024_f32     the benchmark lattice: 1024^2, Mach 0.2 mean flow, state resident in L2
  large_4096_f32    the roofline lattice: 4096^2 with a 128-cell layer, state far larger than L2
  ragged_f16        a lattice of no convenient size in FP16 deviations, type III
  largest_bf16      the 8192^2 lattice of the sweep in BF16 deviations
  source_800x200    the line source of Sec. 4.2 in its channel, to the paper's sample time
  periodic_f64      the FP64 reference format: periodic box, distinct MRT rates, no layer
  compensated_1024  FP32 storage with the compensated collision, the accurate option
  batch_64          64 lattices of mixed sizes (sides 64 to 1024) stepped together
  d3q15_128         the three-dimensional pulse, fields in and out on the host (its interface)
  map_1215          the stability map of Sec. 3.3 over MRT rates, flows and directions
"""
import math
import random

import numpy as np
import torch

from paper_1203_6350_gb300 import lbm, stability
from paper_1203_6350_gb300.batch import Batch

CS = 1.0 / math.sqrt(3.0)


def _solve(name, nx, ny, storage, steps, variant="II", bc="dirichlet", init="pulse", width=20,
           chi_max=0.1, mach=0.0, half=5.0, rates="equal", arithmetic="native", nu=1e-3):
    return dict(kind="solve", name=name, nx=nx, ny=ny, storage=storage, steps=steps,
                variant=variant, bc=bc, init=init, width=width, chi_max=chi_max, mach=mach,
                half=half, rates=rates, arithmetic=arithmetic, nu=nu)


def listed():
    return [
        _solve("small_100_f32", 100, 100, "f32", 300, init="fields", half=3.0),
        dict(kind="history", name="history_200_f32", side=200, every=10, records=52, mach=0.17),
        _solve("flow_1024_f32", 1024, 1024, "f32", 1000, width=64, chi_max=1.0, mach=0.2),
        _solve("large_4096_f32", 4096, 4096, "f32", 200, width=128),
        _solve("ragged_f16", 2050, 1535, "f16dev", 200, variant="III", init="fields", width=37,
               mach=0.1),
        _solve("largest_bf16", 8192, 8192, "bf16dev", 200, width=128),
        dict(kind="source", name="source_800x200", nx=800, ny=200, width=160, steps=2386,
             variant="II", mach=0.0),
        _solve("periodic_f64", 512, 512, "f64", 100, variant="none", bc="periodic", init="fields",
               mach=0.1, rates="mrt"),
        _solve("compensated_1024", 1024, 1024, "f32", 200, width=64, chi_max=0.2, mach=0.2,
               arithmetic="compensated"),
        dict(kind="batch", name="batch_64", count=64, lo=64, hi=1024, steps=200, storage="f32"),
        dict(kind="d3", name="d3q15_128", nx=128, ny=128, nz=128, storage="f32", steps=200,
             variant="II", bc="dirichlet", width=16),
        dict(kind="map", name="map_1215", shear=3, pairs=9, flows=5, directions=3, variants=3,
             nk=127, precision="f32"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["history", "source", "batch", "d3", "map"])
    if kind == "solve":
        storage = rng.choice(["f32", "f32", "f32", "f16dev", "bf16dev", "f64"])
        hi = 768 if storage == "f64" else 6000
        nx, ny = _log_int(rng, 64, hi), _log_int(rng, 64, hi)
        cap = 5e7 if storage == "f64" else 3e9
        steps = min(_log_int(rng, 60, 3000), max(20, int(cap / (nx * ny))))
        # a field that has left the box, or sunk into the roundings of 16 bits, says nothing
        steps = min(steps, 4 * min(nx, ny))
        if storage in ("f16dev", "bf16dev"):
            steps = min(steps, 250, max(20, min(nx, ny) // 2))
        variant = rng.choice(["none", "I", "II", "II", "III", "viscous"])
        width = min(rng.randint(8, 128), (min(nx, ny) - 2) // 2)
        # type I is stable while s + chi <= 2
        chi_max = 0.01 if variant == "I" else math.exp(rng.uniform(math.log(1e-3), 0.0))
        compensated = storage == "f32" and rng.random() < 0.2
        if compensated:
            steps = min(steps, max(20, int(5e8 / (nx * ny))))
        return _solve("", nx, ny, storage, steps, variant=variant,
                      bc=rng.choice(["dirichlet", "dirichlet", "periodic"]),
                      init=rng.choice(["pulse", "fields"]), width=width, chi_max=chi_max,
                      mach=rng.choice([0.0, rng.uniform(0.0, 0.2)]),
                      rates=rng.choice(["equal", "mrt"]),
                      arithmetic="compensated" if compensated else "native") | {"name": "drawn"}
    if kind == "history":
        return dict(kind="history", name="drawn", side=_log_int(rng, 100, 600), every=rng.randint(5, 40),
                    records=rng.randint(10, 60), mach=rng.choice([0.0, 0.17]))
    if kind == "source":
        nx = _log_int(rng, 200, 1600)
        return dict(kind="source", name="drawn", nx=nx, ny=_log_int(rng, 40, 400),
                    width=rng.randint(40, nx // 4), steps=rng.randint(200, 3000),
                    variant=rng.choice(["none", "II", "viscous"]),
                    mach=rng.choice([0.0, 0.17]))
    if kind == "batch":
        return dict(kind="batch", name="drawn", count=_log_int(rng, 8, 96), lo=64,
                    hi=_log_int(rng, 128, 1024), steps=_log_int(rng, 50, 400),
                    storage=rng.choice(["f32", "f32", "f16dev"]))
    if kind == "d3":
        return dict(kind="d3", name="drawn", nx=_log_int(rng, 40, 192), ny=_log_int(rng, 40, 192),
                    nz=_log_int(rng, 40, 192), storage="f32", steps=_log_int(rng, 30, 300),
                    variant=rng.choice(["none", "II", "III"]),
                    bc=rng.choice(["dirichlet", "dirichlet", "periodic"]), width=rng.randint(6, 16))
    return dict(kind="map", name="drawn", shear=rng.randint(1, 3), pairs=rng.randint(1, 9),
                flows=rng.randint(1, 5), directions=rng.randint(1, 3), variants=rng.randint(1, 3),
                nk=rng.choice([31, 63, 100, 127, 200]), precision=rng.choice(["f32", "f32", "f64"]))


# ---------------------------------------------------------------- inputs ----

def _depth(n, width):
    i = np.arange(n)
    return np.clip(width - np.minimum(i, n - 1 - i), 0, width).astype(np.float64)


def _ramp(n, width, chi_max):
    return chi_max * (_depth(n, width) / width) ** 2 if width > 0 else np.zeros(n)


def _orszag(d, width):
    return np.where(d > 0, 3125.0 * (width + 1.0 - d) * d**4 / (256.0 * (width + 1.0) ** 5), 0.0)


def _rate(nu):
    return 1.0 / (3.0 * nu + 0.5)


def _device():
    return "cuda:0" if torch.cuda.is_available() else "cpu"


def _gauss(nx, ny, x0, y0, eps, half):
    x = torch.arange(nx, dtype=torch.float64, device=_device())[None, :]
    y = torch.arange(ny, dtype=torch.float64, device=_device())[:, None]
    return eps * torch.exp(-math.log(2.0) / half**2 * ((x - x0) ** 2 + (y - y0) ** 2))


class _Problem2:
    """One D2Q9 problem: sizes, rates, layer and initial state, from the case and the seed alone."""

    def __init__(self, nx, ny, storage, steps, variant, bc, chi_x, chi_y, s, u0, pulse, fields=False,
                 arithmetic="native", source=None):
        self.nx, self.ny, self.storage, self.steps = nx, ny, storage, steps
        self.variant, self.bc, self.chi_x, self.chi_y = variant, bc, chi_x, chi_y
        self.s, self.u0, self.pulse, self.arithmetic = s, u0, pulse, arithmetic
        self.source, self.n, self.m, self.rho0 = source, 0.5, 0.5, 1.0
        self.fields = fields

    def initial(self):
        """rho - rho0, u_x and u_y of the initial state (FP64): a density pulse on the mean flow, with
        a transverse wave of small amplitude where the program brings fields of its own."""
        eps, half, x0, y0 = self.pulse
        dr = _gauss(self.nx, self.ny, x0, y0, eps, half)
        ux = torch.full_like(dr, self.u0[0])
        uy = torch.full_like(dr, self.u0[1])
        if self.fields:
            x = torch.arange(self.nx, dtype=torch.float64, device=_device())
            uy = uy + 0.2 * eps * torch.sin(2.0 * math.pi / self.nx * x)[None, :]
        return dr, ux, uy

    def make(self):
        lat = lbm.Lattice(self.nx, self.ny, self.storage, self.rho0, self.u0, self.s, self.n, self.m,
                          self.bc)
        lat.set_sponge(self.variant, self.chi_x, self.chi_y)
        if self.source is not None:
            lat.set_source(*self.source)
        if self.arithmetic != "native":
            lat.arithmetic = self.arithmetic
        return lat


def _mrt(s):
    return np.array([s, s, s, 1.5, 1.4, 1.2, 1.2, s, s])


def _problem(case, seed):
    rng = random.Random(seed * 1000003 + 17)
    if case["kind"] == "history":
        side, half = case["side"], max(4.0, case["side"] / 20.0)
        width = min(int(4 * half), side // 2 - 1)
        s = _rate(2e-5)
        chi = 4.0 / s - rng.uniform(0.001, 0.01)
        p = chi * _orszag(_depth(side, width), width)
        c = (side - 1) / 2.0
        return _Problem2(side, side, "f32", case["every"] * case["records"], "II", "dirichlet", p,
                         p.copy(), s, (case["mach"] * CS, 0.0),
                         (rng.uniform(0.8e-3, 1.2e-3), half, c, c))
    if case["kind"] == "source":
        nx, ny, width = case["nx"], case["ny"], case["width"]
        s = _rate(2e-4)
        d = np.clip(np.arange(nx) - (nx - 1 - width), 0, width).astype(np.float64)
        chi_x = {"none": np.zeros(nx), "viscous": d / width,
                 "II": (4.0 / s - 1e-3) * _orszag(d, width)}[case["variant"]]
        return _Problem2(nx, ny, "f32", case["steps"], case["variant"], "channel", chi_x,
                         np.zeros(ny), s, (case["mach"] * CS, 0.02 * CS), (0.0, 1.0, 0.0, 0.0),
                         source=(rng.uniform(0.8e-3, 1.2e-3), 2.0 * math.pi / 100.0,
                                 rng.uniform(0.0, 6.28)))
    nx, ny = case["nx"], case["ny"]
    s = _rate(case["nu"])
    width = case["width"]
    if case["variant"] == "viscous":
        cx, cy = (_depth(n, width) / width for n in (nx, ny))
    else:
        cx, cy = _ramp(nx, width, case["chi_max"]), _ramp(ny, width, case["chi_max"])
    pulse = (rng.uniform(0.8e-3, 1.2e-3), case["half"], rng.uniform(0.3, 0.7) * nx,
             rng.uniform(0.3, 0.7) * ny)
    return _Problem2(nx, ny, case["storage"], case["steps"], case["variant"], case["bc"], cx, cy,
                     _mrt(s) if case["rates"] == "mrt" else s, (case["mach"] * CS, 0.0), pulse,
                     case["init"] == "fields", case["arithmetic"])


def _batch_problems(case, seed):
    rng = random.Random(4711)  # the shapes and layers are the batch's, the fields the seed's
    field = random.Random(seed * 1000003 + 29)
    out = []
    for k in range(case["count"]):
        nx, ny = _log_int(rng, case["lo"], case["hi"]), _log_int(rng, case["lo"], case["hi"])
        variant = ("I", "II", "III")[k % 3]
        width = min(rng.randint(8, 64), (min(nx, ny) - 2) // 2)
        chi = math.exp(rng.uniform(math.log(1e-3), 0.0))
        chi = min(chi, 0.01) if variant == "I" else chi
        out.append(_Problem2(nx, ny, case["storage"], case["steps"], variant, "dirichlet",
                             _ramp(nx, width, chi), _ramp(ny, width, chi), _rate(1e-3),
                             (rng.uniform(0.0, 0.2) * CS, 0.0),
                             (field.uniform(0.8e-3, 1.2e-3), 5.0, field.uniform(0.25, 0.75) * nx,
                              field.uniform(0.25, 0.75) * ny)))
    return out


class _Problem3:
    def __init__(self, case, seed):
        rng = random.Random(seed * 1000003 + 41)
        self.n = (case["nx"], case["ny"], case["nz"])
        self.variant, self.bc, self.steps = case["variant"], case["bc"], case["steps"]
        self.chi = [_ramp(n, min(case["width"], (n - 2) // 2), 0.1) for n in self.n]
        self.s, self.u0 = _rate(1e-3), (0.05, 0.0, 0.02)
        self.eps, self.centre = rng.uniform(0.8e-3, 1.2e-3), [rng.uniform(0.4, 0.6) * n for n in self.n]

    def density(self):
        x, y, z = (np.arange(n) - c for n, c in zip(self.n, self.centre))
        r2 = x[None, None, :] ** 2 + y[None, :, None] ** 2 + z[:, None, None] ** 2
        return 1.0 + self.eps * np.exp(-math.log(2.0) / 25.0 * r2)


def _map_cases(case, seed):
    rng = random.Random(seed * 1000003 + 53)
    shears = [v - rng.uniform(0.0, 5e-4) for v in (1.9, 1.99, 1.999)][: case["shear"]]
    pairs = [(a, b) for a in (1.0, 1.5, None) for b in (1.2, 1.8, None)][: case["pairs"]]
    flows = [0.0, 0.05, 0.1, 0.15, 0.2][: case["flows"]]
    thetas = [0.0, math.pi / 8, math.pi / 4][: case["directions"]]
    names, rows = [], []
    for v in ("II", "I", "III")[: case["variants"]]:
        for s in shears:
            for se, sq in pairs:
                e, q = s if se is None else se, s if sq is None else sq
                for u in flows:
                    for th in thetas:
                        names.append(v)
                        rows.append(stability.case([s, s, s, e, e, q, q, s, s], u_f=(u, 0.0),
                                                   theta=th))
    return names, np.array(rows)


# ---------------------------------------------------------------- a pass ----

def prepare(case, seed):
    kind = case["kind"]
    if kind == "map":
        names, rows = _map_cases(case, seed)
        return dict(kind=kind, names=names, rows=rows, nk=case["nk"], precision=case["precision"])
    if kind == "d3":
        p = _Problem3(case, seed)
        lat = lbm.Lattice3(*p.n, case["storage"], 1.0, p.u0, p.s, bc=p.bc)
        lat.set_sponge(p.variant, *p.chi)
        rho = p.density()
        u = [np.full_like(rho, v) for v in p.u0]
        return dict(kind=kind, lat=lat, rho=rho, u=u, steps=p.steps)
    if kind == "batch":
        ps = _batch_problems(case, seed)
        b = Batch(case["storage"], config=dict(cells=2, steps_per_launch=2, tile=(128, 8)))
        ids, fields = [], []
        for p in ps:
            ids.append(b.add(p.nx, p.ny, p.steps, p.s, p.n, p.m, p.rho0, p.u0, p.bc, p.variant,
                             p.chi_x, p.chi_y))
            dr, ux, uy = p.initial()
            fields.append((dr + p.rho0, ux, uy))
        out = torch.empty((3, sum(p.nx * p.ny for p in ps)), dtype=torch.float64, device=_device())
        return dict(kind=kind, batch=b, ids=ids, fields=fields, out=out, steps=case["steps"],
                    cells=[p.nx * p.ny for p in ps])
    p = _problem(case, seed)
    state = dict(kind=kind, lat=p.make(), p=p)
    if kind == "history":
        state.update(every=case["every"], records=case["records"])
    if p.fields:
        dr, ux, uy = p.initial()
        state["fields"] = (dr + p.rho0, ux, uy)
    return state


def run(state):
    kind = state["kind"]
    if kind == "map":
        return stability.chi_crit(state["names"], state["rows"], nk=state["nk"],
                                  precision=state["precision"], iters=30)
    if kind == "d3":
        lat = state["lat"]
        lat.init_equilibrium(state["rho"], *state["u"])
        lat.step(state["steps"])
        return [f.astype(np.float32) for f in lat.moments()]
    if kind == "batch":
        b, out, at = state["batch"], state["out"], 0
        for i, f in zip(state["ids"], state["fields"]):
            b.init_equilibrium(i, *f)
        b.step(state["steps"])
        for i, n in zip(state["ids"], state["cells"]):
            lbm.lbm_batch_moments(b.b, i, *(out[q, at:at + n].data_ptr() for q in range(3)), 1)
            at += n
        return out.float()
    lat, p = state["lat"], state["p"]
    if "fields" in state:
        lat.init_equilibrium(*state["fields"])
    else:
        lat.init_pulse(*p.pulse)
    if kind == "history":
        rows = [lat.diagnostics()]
        for _ in range(state["records"]):
            lat.step(state["every"])
            rows.append(lat.diagnostics())
        return np.array(rows, dtype=np.float32)
    lat.step(p.steps)
    fields = lat.moments(device=True)
    return list(fields) if p.storage == "f64" else [f.float() for f in fields]


# Floating-point operations of one D2Q9 cell-step (moments, equilibrium, relaxation, transform back)
# and of one D3Q15 cell-step; a 9 x 9 complex eigenproblem by Hessenberg reduction and QR.
_FLOPS2, _FLOPS3, _FLOPS_EIG = 170.0, 320.0, 4.0 * 10.0 * 9**3


def work(case):
    """What a pass cannot do without: the initial fields read once, the results written once, and the
    arithmetic of its steps."""
    kind = case["kind"]
    if kind == "map":
        count = case["shear"] * case["pairs"] * case["flows"] * case["directions"] * case["variants"]
        # the scan to the first unstable value and the halvings after it: about 33 strengths a case
        return {"bytes": count * 16.0 * 8.0, "flops": count * 33.0 * (case["nk"] + 1) * _FLOPS_EIG}
    if kind == "d3":
        cells = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": cells * (4 * 8.0 + 4 * 8.0), "flops": cells * case["steps"] * _FLOPS3}
    if kind == "batch":
        cells = sum(p.nx * p.ny for p in _batch_problems(case, 0))
        return {"bytes": cells * (3 * 8.0 + 3 * 4.0), "flops": cells * case["steps"] * _FLOPS2}
    if kind == "history":
        cells = case["side"] ** 2
        return {"bytes": (case["records"] + 1) * 6 * 4.0,
                "flops": cells * case["every"] * case["records"] * _FLOPS2}
    cells = case["nx"] * case["ny"]
    moved = 3 * (8.0 if case.get("storage") == "f64" else 4.0)
    if case.get("init") == "fields":
        moved += 3 * 8.0
    return {"bytes": cells * moved, "flops": cells * case["steps"] * _FLOPS2}


# ------------------------------------------------- the same in 64 bits ----

_CX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
_CY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
_M = [[1, 1, 1, 1, 1, 1, 1, 1, 1], [0, 1, 0, -1, 0, 1, -1, -1, 1], [0, 0, 1, 0, -1, 1, 1, -1, -1],
      [-4, -1, -1, -1, -1, 2, 2, 2, 2], [4, -2, -2, -2, -2, 1, 1, 1, 1],
      [0, -2, 0, 2, 0, 1, -1, -1, 1], [0, 0, -2, 0, 2, 1, 1, -1, -1],
      [0, 1, -1, 1, -1, 0, 0, 0, 0], [0, 0, 0, 0, 0, 1, -1, 1, -1]]


def _meq(r, jx, jy, linear=False):
    """Moments of the equilibrium (or of its linear part), rows of _M."""
    z = torch.zeros_like(r)
    if linear:
        return torch.stack([r, jx, jy, -2 * r, r, -jx, -jy, z, z])
    xx, yy = jx * jx / r, jy * jy / r
    q = xx + yy
    return torch.stack([r, jx, jy, -2 * r + 3 * q, r - 3 * q, -jx, -jy, xx - yy, jx * jy / r])


class _Exact2:
    """A D2Q9 problem advanced in FP64 on deviations from the far field, in moment space."""

    def __init__(self, p):
        self.p, dev = p, _device()
        self.dev = dev
        self.M = torch.tensor(_M, dtype=torch.float64, device=dev)
        self.Mi = torch.linalg.inv(self.M)
        cx, cy = (torch.tensor(np.asarray(c), dtype=torch.float64, device=dev)
                  for c in (p.chi_x, p.chi_y))
        self.chi = torch.maximum(cx[None, :], cy[:, None])
        if p.variant == "none":
            self.chi = torch.zeros_like(self.chi)
        self.s = torch.tensor(np.broadcast_to(np.asarray(p.s, dtype=np.float64), (9,)).copy(),
                              device=dev)[:, None, None]
        one = torch.ones((1, 1), dtype=torch.float64, device=dev)
        self.base = [p.rho0 * one, p.rho0 * p.u0[0] * one, p.rho0 * p.u0[1] * one]
        self.eq0, self.lin0 = _meq(*self.base), _meq(*self.base, linear=True)
        ux, uy = p.u0
        self.shape = [w * (1 + 3 * (a * ux + b * uy) + 4.5 * (a * ux + b * uy) ** 2
                           - 1.5 * (ux * ux + uy * uy))
                      for w, a, b in zip([4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, _CX, _CY)]
        dr, fx, fy = p.initial()
        rho = p.rho0 + dr
        post = self._mm(self.Mi, _meq(rho, rho * fx, rho * fy) - self.eq0)
        # the state of time 0 is the equilibrium, but for what has entered through the boundary
        g = post
        ny, nx = rho.shape
        for i in range(1, 9):
            if p.bc == "channel":
                if _CX[i] == 1:
                    g[i, :, 0] = self._source(-1) * self.shape[i]
                if _CX[i] == -1:
                    g[i, :, -1] = torch.roll(post[i, :, nx - 2], _CY[i]) if nx > 1 else 0
            elif p.bc == "dirichlet":
                if _CX[i]:
                    g[i, :, 0 if _CX[i] == 1 else -1] = 0
                if _CY[i]:
                    g[i, 0 if _CY[i] == 1 else -1, :] = 0
        self.g, self.time = g, 0

    def _mm(self, a, v):
        return (a @ v.reshape(9, -1)).reshape(v.shape)

    def _source(self, t):
        a, w, ph = self.p.source
        return a * math.sin(w * t + ph)

    def _stream(self, post):
        out = torch.zeros_like(post)
        ny, nx = post.shape[1:]
        bc = self.p.bc
        for i in range(9):
            a, b = _CX[i], _CY[i]
            if bc == "periodic":
                out[i] = torch.roll(post[i], (b, a), (0, 1))
                continue
            src = torch.roll(post[i], b, 0) if bc == "channel" else post[i]
            y0, y1 = (0, 0) if bc == "channel" else (b, b)
            oy = slice(max(y0, 0), ny + min(y0, 0))
            iy = slice(max(-y1, 0), ny + min(-y1, 0))
            out[i, oy, max(a, 0):nx + min(a, 0)] = src[iy, max(-a, 0):nx + min(-a, 0)]
            if bc == "channel" and a == 1:
                out[i, :, 0] = self._source(self.time) * self.shape[i]
            if bc == "channel" and a == -1:
                out[i, :, -1] = src[:, -1]
        return out

    def step(self, n):
        p, chi = self.p, self.chi
        for _ in range(n):
            m = self._mm(self.M, self.g)
            if p.variant == "viscous":
                eq = _meq(self.base[0] + m[0], self.base[1] + m[1], self.base[2] + m[2]) - self.eq0
                s = self.s + (1 - self.s) * chi
                s[:3] = self.s[:3]
                m = m + s * (eq - m)
            else:
                fn, fm = 1 / (1 + p.n * chi), 1 / (1 + p.m * chi)
                # the reference state is the far field: its deviation is zero
                q = [self.base[0] + m[0] * fn, self.base[1] + m[1] * fm, self.base[2] + m[2] * fm]
                eq = _meq(*q) - self.eq0
                if p.variant in ("none", "I"):
                    t = -m
                elif p.variant == "II":
                    t = -eq
                else:
                    t = self.lin0 - _meq(*q, linear=True)
                m = m + self.s * (eq - m) + chi * t
            self.g = self._stream(self._mm(self.Mi, m))
            self.time += 1

    def fields(self):
        m = self._mm(self.M, self.g)[:3]
        rho = self.base[0] + m[0]
        return m[0], (self.base[1] + m[1]) / rho, (self.base[2] + m[2]) / rho

    def sums(self):
        p, (dr, ux, uy) = self.p, self.fields()
        rho = p.rho0 + dr
        e = dr * dr / (6 * p.rho0) + 0.5 * p.rho0 * ((ux - p.u0[0]) ** 2 + (uy - p.u0[1]) ** 2)
        return [float(v.sum()) for v in (dr, rho * ux - p.rho0 * p.u0[0], rho * uy - p.rho0 * p.u0[1],
                                         e, dr * dr, (~torch.isfinite(rho + ux + uy)).double())]


def _exact3(case, seed):
    p, dev = _Problem3(case, seed), _device()
    c = [(0, 0, 0)] + [tuple(sg if k == ax else 0 for k in range(3)) for ax in range(3) for sg in (1, -1)]
    c += [(a, b, d) for d in (1, -1) for b in (1, -1) for a in (1, -1)]
    w = [2 / 9] + [1 / 9] * 6 + [1 / 72] * 8

    def eq(r, j, linear=False):
        out = []
        for ci, wi in zip(c, w):
            cj = sum(a * b for a, b in zip(ci, j) if a) if any(ci) else torch.zeros_like(r)
            if linear:
                out.append(wi * (r + 3 * cj))
            else:
                out.append(wi * (r + 3 * cj + (4.5 * cj * cj - 1.5 * sum(b * b for b in j)) / r))
        return torch.stack(out)

    rho = torch.tensor(p.density(), device=dev)
    one = torch.ones((1, 1, 1), dtype=torch.float64, device=dev)
    j0 = [v * one for v in p.u0]
    f0, l0 = eq(one, j0), eq(one, j0, True)
    g = eq(rho, [v * rho for v in p.u0]) - f0
    cx, cy, cz = (torch.tensor(v, device=dev) for v in p.chi)
    chi = torch.maximum(torch.maximum(cx[None, None, :], cy[None, :, None]), cz[:, None, None])
    if p.variant == "none":
        chi = torch.zeros_like(chi)
    f = 1 / (1 + 0.5 * chi)
    dims = rho.shape

    def wall(v, ci, i):  # nothing but the far field enters through a wall
        for ax, a in zip((2, 1, 0), ci):
            if a:
                v[i].select(ax, 0 if a == 1 else dims[ax] - 1).zero_()

    for i, ci in enumerate(c):
        if p.bc == "dirichlet":
            wall(g, ci, i)
    for _ in range(p.steps):
        r = g.sum(0)
        j = [sum(ci[k] * g[i] for i, ci in enumerate(c) if ci[k]) for k in range(3)]
        rs, js = 1 + r * f, [b + v * f for b, v in zip(j0, j)]
        es = eq(rs, js) - f0
        post = g + p.s * (es - g)
        if p.variant == "II":
            post -= chi * es
        elif p.variant == "III":
            post += chi * (l0 - eq(rs, js, True))
        for i, ci in enumerate(c):
            g[i] = torch.roll(post[i], (ci[2], ci[1], ci[0]), (0, 1, 2))
            if p.bc == "dirichlet":
                wall(g, ci, i)
    r = g.sum(0)
    j = [sum(ci[k] * g[i] for i, ci in enumerate(c) if ci[k]) for k in range(3)]
    return [r.cpu().numpy()] + [((b + v) / (1 + r)).cpu().numpy() for b, v in zip(j0, j)]


def _growth(rows, names, chi, nk):
    """Largest |lambda| of the linearised step over the wavenumbers, for each row at its own chi."""
    M = np.array(_M, dtype=np.float64)
    Mi = np.linalg.inv(M)
    out = np.empty(len(rows))
    for q, (row, name) in enumerate(zip(rows, names)):
        s, n, m, ux, uy, th = row[:9], row[9], row[10], row[11], row[12], row[13]
        uu = ux * ux + uy * uy
        Q, L = np.zeros((9, 9)), np.zeros((9, 9))
        Q[:, 0] = [1, 0, 0, -2 - 3 * uu, 1 + 3 * uu, 0, 0, -(ux * ux - uy * uy), -ux * uy]
        Q[:, 1] = [0, 1, 0, 6 * ux, -6 * ux, -1, 0, 2 * ux, uy]
        Q[:, 2] = [0, 0, 1, 6 * uy, -6 * uy, 0, -1, -2 * uy, ux]
        L[:, 0], L[:, 1], L[:, 2] = ([1, 0, 0, -2, 1, 0, 0, 0, 0], [0, 1, 0, 0, 0, -1, 0, 0, 0],
                                     [0, 0, 1, 0, 0, 0, -1, 0, 0])
        scale = np.ones(9)
        scale[0], scale[1], scale[2] = 1 / (1 + n * chi[q]), 1 / (1 + m * chi[q]), 1 / (1 + m * chi[q])
        Q, L = Q * scale, L * scale
        A = np.eye(9) - np.diag(s) + np.diag(s) @ Q
        A -= chi[q] * {"I": np.eye(9), "II": Q, "III": L}[name]
        J = Mi @ A @ M
        k = np.pi * np.arange(nk + 1) / nk
        ph = np.exp(-1j * k[:, None] * (np.cos(th) * np.array(_CX) + np.sin(th) * np.array(_CY)))
        out[q] = np.abs(np.linalg.eigvals(ph[:, :, None] * J)).max()
    return out


def _exact_map(case, seed):
    names, rows = _map_cases(case, seed)
    if len(rows) * (case["nk"] + 1) * 40 > 5e5:
        return None  # minutes of eigenproblems
    limit = 1.0 + (1e-9 if case["precision"] == "f64" else 1e-5)
    out = []
    for name, row in zip(names, rows):
        def unstable(chi):
            return _growth([row], [name], [chi], case["nk"])[0] > limit

        if unstable(0.0):
            out.append(-math.inf)
            continue
        grid = [8.0 * g / 16 for g in range(17)]
        first = next((g for g in range(1, 17) if unstable(grid[g])), None)
        if first is None:
            out.append(math.inf)
            continue
        a, b = grid[first - 1], grid[first]
        for _ in range(30):
            mid = 0.5 * (a + b)
            a, b = (a, mid) if unstable(mid) else (mid, b)
        out.append(0.5 * (a + b))
    return np.array(out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "map":
        return _exact_map(case, seed)
    if kind == "d3":
        return _exact3(case, seed)
    if kind == "batch":
        if case["count"] * case["steps"] > 16000:
            return None  # one lattice after another
        fields = []
        for p in _batch_problems(case, seed):
            e = _Exact2(p)
            e.step(p.steps)
            fields.append(torch.stack([f.reshape(-1) for f in e.fields()]))
        return torch.cat(fields, dim=1)
    p = _problem(case, seed)
    if p.nx * p.ny * p.steps > 2e10:
        return None
    e = _Exact2(p)
    if kind == "history":
        rows = [e.sums()]
        for _ in range(case["records"]):
            e.step(case["every"])
            rows.append(e.sums())
        return np.array(rows)
    e.step(p.steps)
    return list(e.fields())
