"""Performance cases of the HBGK library: what its users run, through its public entry points.

A case is a dict of plain values. Its "kind" names the call that is measured:

  steps    a lattice advanced by `steps` time steps, then its diagnostics (reduce), its density and
           velocity (moments) and its populations (checkpoint or coupling), read into device buffers
  host     a whole solve from host data: porosity field in, start from rest, steps, diagnostics,
           density and velocity out, all host arrays
  adjoint  value and porosity gradient of the outflow flux on a lattice the program keeps
  autograd the same through the torch.autograd.Function, as one iteration of a design loop calls it
  memory   the relaxation history of the Darcy law with memory (one diagnostics record per step)
  serve    a batch of solve requests through the continuous-batching server

Fields are periodic matrices of spheres (one per cell of about `period` lattice cells) whose radius
and position are drawn from the seed; flows start from a uniform velocity drawn from the seed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2310_14746_gb300 as hb
from paper_2310_14746_gb300 import autograd, workloads
from paper_2310_14746_gb300.serving import Server

STORAGE = {"f64": hb.HLBM_F64, "f32": hb.HLBM_F32, "f16": hb.HLBM_F16DEV, "bf16": hb.HLBM_BF16DEV}
BYTES = {"f64": 8, "f32": 4, "f16": 2, "bf16": 2}
FLOPS = {9: 110, 19: 250}  # floating-point operations of one cell update, about
SERVE_EDGES = (32, 48, 64, 96)


def _steps(name, nx, ny, nz, steps, q=19, storage="f32", pattern="two", form="shift", walls="", field="spheres",
           oblique=False):
    return {"name": name, "kind": "steps", "q": q, "nx": nx, "ny": ny, "nz": nz, "steps": steps, "storage": storage,
            "pattern": pattern, "form": form, "walls": walls, "field": field, "oblique": oblique}


def listed():
    return [
        # the Brinkman channel of the validation study: the smallest lattice in use, launches and latency
        _steps("channel_f32", 64, 32, 1, 1000, q=9, walls="y", field="uniform"),
        # the same in the 64-bit policy that the study compares with
        _steps("channel_f64", 64, 32, 1, 500, q=9, storage="f64", walls="y", field="uniform"),
        # one check interval of the resolved-sphere permeability study: a small box with voxel obstacles
        _steps("pore_32_f32", 32, 32, 32, 100, field="solid"),
        # one check interval of the main benchmark: FP32 at 256^3
        _steps("sphere_256_f32", 256, 256, 256, 100),
        # reduced-precision storage at 384^3, the largest lattice of the benchmark
        _steps("sphere_384_f16", 384, 384, 384, 60, storage="f16"),
        # the memory-saving in-place pattern in BF16
        _steps("inplace_192_bf16", 192, 192, 192, 100, storage="bf16", pattern="aa"),
        # a duct with walls, the drag form and a force along all axes, on sizes that divide by nothing
        _steps("duct_drag_f32", 150, 101, 67, 100, form="drag", walls="y", oblique=True),
        # a solve from host arrays, as a script calls it
        {"name": "host_160_f32", "kind": "host", "n": 160, "steps": 100, "storage": "f32"},
        # the flux gradient at 128^3 with recomputation every 45 steps, a section of the 2000-step run
        {"name": "adjoint_128_f32", "kind": "adjoint", "nx": 128, "ny": 128, "nz": 128, "steps": 180, "every": 45,
         "storage": "f32", "walls": ""},
        # one iteration of a design loop on a small box, through torch.autograd
        {"name": "autograd_48_f32", "kind": "autograd", "nx": 48, "ny": 48, "nz": 48, "steps": 90, "every": 45,
         "storage": "f32", "walls": ""},
        # the relaxation history of one sphere cell
        {"name": "memory_64_f32", "kind": "memory", "n": 64, "steps": 200, "storage": "f32"},
        # a mixed batch of permeability requests on the FP16 server
        {"name": "serve_f16", "kind": "serve", "requests": 12, "steps": 400, "storage": "f16", "max_edge": 96},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))))


def draw(rng):
    kind = rng.choice(["steps"] * 10 + ["host", "adjoint", "autograd", "memory", "serve"])
    if kind == "steps":
        q = 9 if rng.random() < 0.15 else 19
        storage = rng.choice(["f32", "f32", "f16", "bf16", "f64"])
        pattern = "aa" if rng.random() < 0.2 else "two"
        form = rng.choice(["shift", "shift", "shift", "drag", "tensor"])
        field = rng.choice(["spheres", "spheres", "spheres", "solid"])
        walls = rng.choice(["", "", "", "y"]) if q == 9 else rng.choice(["", "", "", "", "y", "yz"])
        if q == 9:
            nx, ny, nz = _log_int(rng, 32, 2048), _log_int(rng, 24, 1536), 1
        else:
            base = _log_int(rng, 24, 160 if storage == "f64" else 288)
            nx, ny, nz = (max(16, int(base * rng.uniform(0.7, 1.3))) for _ in range(3))
            if rng.random() < 0.5:  # common sizes: multiples of 8
                nx, ny, nz = (max(16, 8 * round(v / 8)) for v in (nx, ny, nz))
        cost = nx * ny * nz * q * (2 * BYTES[storage] if storage != "f64" else 128)
        most = max(8, min(400, int(6e10 / cost)))
        return {k: v for k, v in _steps("", nx, ny, nz, _log_int(rng, min(20, most), most), q, storage, pattern, form,
                                        walls, field, rng.random() < 0.4).items() if k != "name"}
    if kind == "host":
        return {"kind": kind, "n": _log_int(rng, 32, 224), "steps": rng.randint(60, 150),
                "storage": rng.choice(["f32", "f32", "f16"])}
    if kind in ("adjoint", "autograd"):
        base = _log_int(rng, 24, 128 if kind == "adjoint" else 80)
        nx, ny, nz = (max(16, int(base * rng.uniform(0.8, 1.2))) for _ in range(3))
        return {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "steps": rng.randint(45, 150), "every": rng.choice([15, 30, 45]),
                "storage": rng.choice(["f32", "f32", "f16"]), "walls": rng.choice(["", "", "y"])}
    if kind == "memory":
        return {"kind": kind, "n": _log_int(rng, 24, 128), "steps": rng.randint(100, 300), "storage": "f32"}
    return {"kind": kind, "requests": rng.randint(4, 16), "steps": 100 * rng.randint(2, 5),
            "storage": rng.choice(["f16", "f16", "f32", "bf16"]), "max_edge": rng.choice([48, 64, 96])}


# ---- inputs -----------------------------------------------------------------------------------------

def _gen(seed, salt=0):
    return np.random.default_rng([int(seed) & 0x7fffffff, salt])


def _distance(shape, period, ratio, shift):
    """Distance of every cell to the surface of the nearest sphere (float32 [nz, ny, nx] on the GPU)."""
    total = None
    for axis, n in zip((2, 1, 0), shape[::-1]):  # x, y, z
        if n == 1:
            continue
        p = n / max(1, round(n / period))
        t = torch.remainder(torch.arange(n, device="cuda", dtype=torch.float32) + 0.5 + float(shift[axis]), p) - 0.5 * p
        t = (t * t).reshape([-1 if a == axis else 1 for a in range(3)])
        total = t if total is None else total + t
    return (torch.sqrt(total) - ratio * min(period, *[n for n in shape if n > 1])).expand(shape)


def _field(shape, rng, period=32.0):
    """Smoothed sphere matrix varpi in [0, 1] (transition width 2 cells)."""
    s = _distance(shape, period, rng.uniform(0.2, 0.4), rng.uniform(0, period, 3))
    return (0.5 * (1 + torch.sin(math.pi * torch.clamp(s / 2, -0.5, 0.5)))).clamp(0, 1).contiguous()


def _bc(case):
    return tuple(1 if a in case.get("walls", "") else 0 for a in "xyz")


def _problem(case, seed):
    """Everything that defines the flow: shape, tau, F, u0, porosity (scalar or tensor), solid cells."""
    rng = _gen(seed)
    shape = (case["nz"], case["ny"], case["nx"])
    p = {"shape": shape, "bc": _bc(case), "tau": 0.8 if case["q"] == 9 else 0.6, "solid": None, "varpi3": None}
    p["F"] = (1e-6, -4e-7, 3e-7 if case["q"] == 19 else 0.0) if case["oblique"] else (1e-6, 0.0, 0.0)
    p["u0"] = tuple(float(v) for v in rng.uniform(0.002, 0.01, 3) * (1, 0.5, 0.5 if case["q"] == 19 else 0))
    if case["field"] == "uniform":
        p["varpi"] = torch.full(shape, float(rng.uniform(0.85, 0.95)), device="cuda")
    elif case["field"] == "solid":
        s = _distance(shape, 32.0, rng.uniform(0.2, 0.35), rng.uniform(0, 32, 3))
        p["solid"] = (s < 0).to(torch.uint8).contiguous()
        p["varpi"] = torch.ones(shape, device="cuda")
    else:
        p["varpi"] = _field(shape, rng)
    if case["form"] == "tensor":
        k = [float(v) for v in rng.uniform(0.5, 1.0, 3)]
        p["varpi3"] = torch.stack([1 - k[a] * (1 - p["varpi"]) for a in range(3)]).contiguous()
    return p


def _lattice(q, p, storage, pattern="two", form="shift"):
    nz, ny, nx = p["shape"]
    lat = hb.Lattice(q, nx, ny, nz, STORAGE[storage], hb.HLBM_AA if pattern == "aa" else hb.HLBM_TWO_LATTICE)
    lat.set_relaxation(p["tau"])
    lat.set_force(*p["F"])
    for a, b in enumerate(p["bc"]):
        lat.set_boundary(a, hb.HLBM_HALFWAY_BOUNCE_BACK if b else hb.HLBM_PERIODIC)
    lat.set_porosity(p["varpi"])
    if form == "drag":
        lat.set_homogenization(hb.HLBM_HOMOG_DRAG)
    if form == "tensor":
        lat.set_porosity_tensor(p["varpi3"])
    if p["solid"] is not None:
        lat.set_solid_mask(p["solid"])
    lat.init_equilibrium(1.0, p["u0"])
    return lat


def _flow(case, seed):
    """The shift-form problem of the adjoint, autograd and host kinds (start from rest)."""
    c = dict(case, q=19, field="spheres", form="shift", oblique=False)
    if "n" in case:
        c.update(nx=case["n"], ny=case["n"], nz=case["n"], walls="")
    p = _problem(c, seed)
    p["u0"] = (0.0, 0.0, 0.0)
    return p


def _requests(case, seed):
    rng = _gen(seed, 7)
    size = np.random.default_rng([case["requests"], case["max_edge"]])  # the mix of sizes is the case's
    edges = [e for e in SERVE_EDGES if e <= case["max_edge"]]
    out = []
    for k in range(case["requests"]):
        n = int(size.choice(edges))
        out.append(_field((n, n, n), rng, period=float(size.choice([16, 32]))).cpu().numpy())
    return out


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case}
    if kind == "steps":
        p = _problem(case, seed)
        st["lat"] = _lattice(case["q"], p, case["storage"], case["pattern"], case["form"])
        real = torch.float64 if case["storage"] == "f64" else torch.float32
        st["rho"] = torch.empty(p["shape"], dtype=real, device="cuda")
        st["u"] = torch.empty((3,) + p["shape"], dtype=real, device="cuda")
        st["f"] = torch.empty((case["q"],) + p["shape"], dtype=torch.float64, device="cuda")
    elif kind == "host":
        p = _flow(case, seed)
        st["varpi"] = p["varpi"].cpu().numpy()
        st["lat"] = _lattice(19, p, case["storage"])
    elif kind == "adjoint":
        p = _flow(case, seed)
        st["lat"] = _lattice(19, p, case["storage"])
        st["grad"] = torch.empty(p["shape"], dtype=torch.float32, device="cuda")
    elif kind == "autograd":
        p = _flow(case, seed)
        st["varpi"] = p["varpi"]
        st["cfg"] = {"tau": p["tau"], "F": p["F"], "nsteps": case["steps"], "ckpt_every": case["every"], "bc": p["bc"],
                     "storage": STORAGE[case["storage"]]}
    elif kind == "memory":
        p = _flow(case, seed)
        st["varpi"] = p["varpi"].cpu().numpy()
    else:
        st["server"] = Server(8 << 30, STORAGE[case["storage"]], 100)
        st["fields"] = _requests(case, seed)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "steps":
        lat = st["lat"]
        lat.step(case["steps"])
        stats = lat.reduce()
        if case["storage"] == "f64":
            hb.hlbm_moments_f64(lat.h, st["rho"], st["u"])
        else:
            hb.hlbm_moments(lat.h, st["rho"], st["u"])
        hb.hlbm_get_populations(lat.h, st["f"])
        return {"f": st["f"], "rho": st["rho"], "stats": stats, "u": st["u"]}
    if kind == "host":
        lat = st["lat"]
        lat.set_porosity(st["varpi"])
        lat.init_equilibrium()
        lat.step(case["steps"])
        stats = lat.reduce()
        rho, u = lat.moments()
        return {"rho": rho, "stats": stats, "u": u}
    if kind == "adjoint":
        J, grad = st["lat"].adjoint_flux_grad(case["steps"], case["every"], None, st["grad"])
        return {"J": J, "grad": grad}
    if kind == "autograd":
        J, grad = autograd.flux_and_grad(st["varpi"], **st["cfg"])
        return {"J": J, "grad": grad}
    if kind == "memory":
        return {"A": workloads.memory_kernel(st["varpi"], 0.6, case["steps"], storage=STORAGE[case["storage"]])}
    # an interval is 100 steps; the tolerance is out of reach, so every solve runs its full length
    srv = st["server"]
    ids = [srv.submit(v, tol=1e-9, max_steps=case["steps"], want_u=True) for v in st["fields"]]
    got = {r["id"]: r for r in srv.run_until_idle()}
    out = {k: np.array([got[i][k] for i in ids]) for k in ("k_app", "mass", "max_u", "status", "steps")}
    return dict(out, u=[got[i]["u"] for i in ids])


def work(case):
    """One pass: the state, field and forces read once, everything handed back written once."""
    kind = case["kind"]
    if kind == "serve":
        size = np.random.default_rng([case["requests"], case["max_edge"]])
        edges = [e for e in SERVE_EDGES if e <= case["max_edge"]]
        cells = 0
        for _ in range(case["requests"]):
            cells += int(size.choice(edges)) ** 3
            size.choice([16, 32])
        return {"bytes": cells * (4 + 12), "flops": cells * case["steps"] * FLOPS[19]}
    n = case["n"] ** 3 if "n" in case else case["nx"] * case["ny"] * case["nz"]
    b = BYTES[case["storage"]]
    q = case.get("q", 19)
    flops = n * case["steps"] * FLOPS[q]
    if kind == "steps":
        real = 8 if case["storage"] == "f64" else 4
        field = 12 if case["form"] == "tensor" else 4
        links = 1 if case["field"] == "solid" else 0
        return {"bytes": n * (2 * q * b + field + links + 4 * real + 8 * q), "flops": flops}
    if kind == "host":
        return {"bytes": n * (4 + 16), "flops": flops}
    if kind == "adjoint":  # the state goes from the first to the last step; a reverse step costs about two forward ones
        return {"bytes": n * (8 + 2 * q * b), "flops": 3 * flops}
    if kind == "autograd":
        return {"bytes": 8 * n, "flops": 3 * flops}
    return {"bytes": 4 * n + 8 * case["steps"], "flops": flops}


# ---- the same in 64 bits, with torch alone ------------------------------------------------------------

_C9 = [(0, 0, 0), (1, 0, 0), (0, 1, 0), (-1, 0, 0), (0, -1, 0), (1, 1, 0), (-1, 1, 0), (-1, -1, 0), (1, -1, 0)]
_C19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0), (1, -1, 0),
        (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]


class _Exact:
    """Plain HBGK steps on a list of q float64 tensors [nz, ny, nx] (full populations)."""

    def __init__(self, q, p, form="shift"):
        self.c = _C9 if q == 9 else _C19
        n2 = [sum(v * v for v in c) for c in self.c]
        self.w = [{0: 4 / 9, 1: 1 / 9, 2: 1 / 36}[k] if q == 9 else {0: 1 / 3, 1: 1 / 18, 2: 1 / 36}[k] for k in n2]
        self.opp = [self.c.index(tuple(-v for v in c)) for c in self.c]
        self.tau, self.F, self.bc, self.form, self.shape = p["tau"], p["F"], p["bc"], form, p["shape"]
        self.varpi = p["varpi"].double()
        self.varpi3 = None if p["varpi3"] is None else [v.double() for v in p["varpi3"]]
        self.solid = None if p["solid"] is None else p["solid"].bool()
        self.source_solid = None
        if self.solid is not None:
            self.source_solid = [self._shift(self.solid, c) for c in self.c]

    def start(self, u0):
        uu = sum(v * v for v in u0)
        f = []
        for c, w in zip(self.c, self.w):
            cu = sum(a * b for a, b in zip(c, u0))
            f.append(torch.full(self.shape, w * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * uu), dtype=torch.float64, device="cuda"))
        if self.solid is not None:
            f = [torch.where(self.solid, w, v) for w, v in zip(self.w, f)]
        return f

    @staticmethod
    def _shift(v, c):
        s, d = zip(*[(c[2 - a], a) for a in range(3) if c[2 - a]]) if any(c) else ((), ())
        return torch.roll(v, s, d) if s else v

    def stream(self, f):
        g = []
        for i, c in enumerate(self.c):
            v = self._shift(f[i], c)
            back = f[self.opp[i]]
            for a in range(3):
                if self.bc[a] and c[a]:
                    n = self.shape[2 - a]
                    at = torch.arange(n, device="cuda") == (0 if c[a] > 0 else n - 1)
                    v = torch.where(at.reshape([-1 if d == 2 - a else 1 for d in range(3)]), back, v)
            if self.solid is not None and i:
                wall = self.source_solid[i]
                for a in range(3):
                    if self.bc[a] and c[a]:
                        n = self.shape[2 - a]
                        at = torch.arange(n, device="cuda") == (0 if c[a] > 0 else n - 1)
                        wall = wall & ~at.reshape([-1 if d == 2 - a else 1 for d in range(3)])
                v = torch.where(wall, back, v)
            g.append(v)
        return g

    def moments(self, g, varpi=None):
        rho = sum(g)
        h = 1.0
        if self.form == "drag":
            h = 1 / (1 + 0.5 * (1 - self.varpi) / self.tau)
        u = []
        for a in range(3):
            j = sum(c[a] * v for c, v in zip(self.c, g) if c[a])
            u.append((j + 0.5 * self.F[a]) / rho * h)
        return rho, u

    def collide(self, g, varpi=None):
        vp = self.varpi if varpi is None else varpi
        rho, u = self.moments(g)
        om, guo = 1 / self.tau, 1 - 0.5 / self.tau
        F = self.F
        if self.form == "drag":
            lam = (1 - vp) * om
            F = [self.F[a] - lam * rho * u[a] for a in range(3)]
            v = u
        elif self.form == "tensor":
            v = [self.varpi3[a] * u[a] for a in range(3)]
        else:
            v = [vp * u[a] for a in range(3)]
        vv = v[0] * v[0] + v[1] * v[1] + v[2] * v[2]
        uF = u[0] * F[0] + u[1] * F[1] + u[2] * F[2]
        base, src = 1 - 1.5 * vv, -3 * uF
        out = []
        for c, w, gi in zip(self.c, self.w, g):
            if not any(c):
                out.append(gi - om * (gi - w * rho * base) + guo * w * src)
                continue
            cv = sum(a * b for a, b in zip(c, v) if a)
            cu = sum(a * b for a, b in zip(c, u) if a)
            cF = sum(a * b for a, b in zip(c, F) if a)
            out.append(gi - om * (gi - w * rho * (base + 3 * cv + 4.5 * cv * cv)) + guo * w * (src + 3 * cF + 9 * cu * cF))
        return out

    def step(self, f):
        new = self.collide(self.stream(f))
        return new if self.solid is None else [torch.where(self.solid, a, b) for a, b in zip(f, new)]

    def observe(self, f):
        rho, u = self.moments(self.stream(f))
        if self.solid is not None:
            rho, u = torch.where(self.solid, 1.0, rho), [torch.where(self.solid, 0.0, v) for v in u]
        return rho, torch.stack(u)

    def stats(self, rho, u):
        jx = float((rho * u[0]).sum()) if self.solid is None else float((rho * u[0])[~self.solid].sum())
        return {"k_app": (self.tau - 0.5) / 3 * jx / rho.numel() / self.F[0], "mass": float(rho.sum()), "max_du": None,
                "max_u": float(u.abs().max()), "mom_x": jx, "mom_y": None, "mom_z": None, "plane_flux": None, "step": None}


def _exact_gradient(case, p):
    """J and dJ/dvarpi by torch's reverse mode, one step at a time from kept states."""
    ex = _Exact(19, p)
    states = [torch.stack(ex.start(p["u0"]))]
    with torch.no_grad():
        for _ in range(case["steps"]):
            states.append(torch.stack(ex.step(list(states[-1]))))
    last = states[-1].requires_grad_(True)
    plane = p["shape"][2] - 1
    jx = sum(c[0] * v[:, :, plane] for c, v in zip(ex.c, ex.stream(list(last))) if c[0])
    J = (jx + 0.5 * p["F"][0]).sum()
    lam = torch.autograd.grad(J, last)[0]
    grad = torch.zeros(p["shape"], dtype=torch.float64, device="cuda")
    for s in range(case["steps"] - 1, -1, -1):
        f = states[s].detach().requires_grad_(True)
        vp = ex.varpi.detach().requires_grad_(True)
        new = torch.stack(ex.collide(ex.stream(list(f)), vp))
        lam, gv = torch.autograd.grad(new, (f, vp), lam)
        grad += gv
        states.pop()
    return {"J": float(J.detach()), "grad": grad}


def exact(case, seed):
    kind = case["kind"]
    if kind == "steps":
        p = _problem(case, seed)
        ex = _Exact(case["q"], p, case["form"])
        f = ex.start(p["u0"])
        for _ in range(case["steps"]):
            f = ex.step(f)
        rho, u = ex.observe(f)
        return {"f": torch.stack(f), "rho": rho, "stats": ex.stats(rho, u), "u": u}
    if kind == "host":
        p = _flow(case, seed)
        ex = _Exact(19, p)
        f = ex.start(p["u0"])
        for _ in range(case["steps"]):
            f = ex.step(f)
        rho, u = ex.observe(f)
        return {"rho": rho, "stats": ex.stats(rho, u), "u": u}
    if kind in ("adjoint", "autograd"):
        return _exact_gradient(case, _flow(case, seed))
    if kind == "memory":
        p = dict(_flow(case, seed), F=(0.0, 0.0, 0.0), tau=0.6)
        ex = _Exact(19, p)
        f = ex.start((1e-4, 0.0, 0.0))
        out = []
        for s in range(case["steps"]):
            g = ex.stream(f)
            out.append(sum(c[0] * v.sum() for c, v in zip(ex.c, g) if c[0]) / g[0].numel() / 1e-4)
            f = ex.collide(g)
        return {"A": torch.stack(out)}
    out = {"k_app": [], "mass": [], "max_u": [], "status": None, "steps": None, "u": []}
    for v in _requests(case, seed):
        p = {"shape": v.shape, "bc": (0, 0, 0), "tau": 0.6, "F": (1e-6, 0.0, 0.0), "varpi": torch.from_numpy(v).cuda(),
             "varpi3": None, "solid": None}
        ex = _Exact(19, p)
        f = ex.start((0.0, 0.0, 0.0))
        for _ in range(case["steps"]):
            f = ex.step(f)
        rho, u = ex.observe(f)
        s = ex.stats(rho, u)
        for k in ("k_app", "mass", "max_u"):
            out[k].append(s[k])
        out["u"].append(u)
    return {k: np.array(v) if k in ("k_app", "mass", "max_u") else v for k, v in out.items()}
