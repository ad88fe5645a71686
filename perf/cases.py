"""Performance cases of the framework: the calls a user's program makes, from the smallest
lattice of the paper's experiments to the full-size benchmark, through the public wrappers
(`lattice.Lattice`, `lattice.run`, `batch.Batch`, `capi.lbm_run_host`).

Kinds of case:
  run    one lattice: initial fields -> n steps -> (rho, u), optionally with fused diagnostics
         (read back) and fullway bounce-back walls at the two ends of x
  grad   one lattice: the differentiable run, a loss on the final fields and its backward pass
  batch  independent domains of uneven size, theta and tau advanced together
  host   the end-to-end call on page-locked host memory
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2602_21242_gb300 import capi, flows
from paper_2602_21242_gb300.batch import Batch
from paper_2602_21242_gb300.lattice import Lattice, run as run_lattice, tau_from_nu

THIRD = 1.0 / 3.0
# arithmetic operations of one node update by the method's formulas (adds, products and fused
# multiply-adds each counted once), by model
OPS = {"lbgk": 60, "oreg": 93, "partial": 103, "complete": 123, "complete_neq": 120}


def _case(kind, nx, ny, steps, prec="f64", model="complete", theta=THIRD, nu=0.005, flow="vortex", U=0.1, **more):
    return {"kind": kind, "nx": nx, "ny": ny, "steps": steps, "prec": prec, "model": model, "theta": theta, "nu": nu,
            "flow": flow, "U": U, **more}


def listed():
    return [
        # the paper's decay check: the smallest two-dimensional lattice, advanced over its whole run
        dict(_case("run", 64, 64, 1000, nu=0.01, flow="taylor_green", U=0.0), name="taylor_green_64_f64"),
        # the paper's shocktube (Sec. 5.2): one row between two bounce-back walls, fluid at rest along it
        dict(_case("run", 800, 1, 400, model="partial", theta=0.4, nu=1e-9, flow="shocktube", U=0.0, walls=True),
             name="shocktube_800x1_f64"),
        # the paper's shear layer (Sec. 5.3) at its middle grid, mass and momentum watched
        dict(_case("run", 256, 256, 500, model="oreg", theta=0.4, nu=3.4e-4, flow="shear_layer", U=0.04, diag=50),
             name="shear_layer_256_f64"),
        # the bandwidth benchmark in the paper's precision, diagnostics every step
        dict(_case("run", 4096, 4096, 10, flow="shear_wave", diag=1), name="shear_wave_4096_f64"),
        # the fast form of FP64 storage, on a grid that is no multiple of any tile
        dict(_case("run", 1531, 1277, 40, prec="f64df", theta=0.4), name="vortex_1531x1277_f64df"),
        # FP32 storage on an ordinary grid with odd sides
        dict(_case("run", 601, 487, 200, prec="f32", model="complete", theta=0.3, nu=1e-3), name="vortex_601x487_f32"),
        # the bandwidth benchmark in FP32 storage, and its LBGK in FP16 storage on a ragged width
        dict(_case("run", 4096, 4096, 40, prec="f32", flow="shear_wave", diag=10), name="shear_wave_4096_f32"),
        dict(_case("run", 4090, 3072, 40, prec="f16", flow="shear_layer", theta=0.3, nu=1e-3), name="shear_layer_4090x3072_f16"),
        # the batched workload: 256 uneven Taylor-Green domains, FP32 storage
        dict(_case("batch", 64, 512, 50, prec="f32", flow="taylor_green", count=256), name="batch_256_f32"),
        # gradients of a misfit of the final fields, with checkpoints: FP64, and FP32 at the size of the
        # differentiation benchmark
        dict(_case("grad", 384, 384, 100, nu=0.01, U=0.0, every=25), name="gradient_384_f64"),
        dict(_case("grad", 1024, 1024, 100, prec="f32", nu=0.01, U=0.0, every=50), name="gradient_1024_f32"),
        # host arrays in, host arrays out
        dict(_case("host", 2048, 2048, 10, flow="shear_wave"), name="host_2048_f64"),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["run", "run", "run", "run", "grad", "batch", "host"])
    prec = rng.choice({"run": ["f64", "f64", "f32", "f16", "f64df"], "grad": ["f64", "f32"], "batch": ["f32", "f32", "f64"],
                       "host": ["f64", "f64", "f32"]}[kind])
    model = rng.choice(["lbgk", "oreg", "partial", "complete", "complete", "complete_neq"])
    theta = rng.choice([THIRD, 0.3, 0.35, 0.4])
    nu = round(math.exp(rng.uniform(math.log(0.004), math.log(0.02))), 5)
    flow = rng.choice(["vortex", "vortex", "shear_wave", "shear_layer", "taylor_green"])
    U = rng.choice([0.0, 0.05, 0.1]) if flow != "shear_layer" else 0.05
    if kind == "batch":
        return _case(kind, rng.randint(24, 96), rng.randint(128, 400), log(10, 60), prec, model, THIRD, 0.01,
                     "taylor_green", 0.0, count=log(4, 64))
    if kind == "grad":
        n = log(20, 100)
        return _case(kind, log(32, 600), log(32, 600), n, prec, model, theta, nu, "vortex", 0.0, every=rng.randint(5, n))
    if kind == "host":
        return _case(kind, log(64, 2000), log(64, 2000), log(5, 20), prec, model, theta, nu, flow, U)
    nx, ny = log(16, 4096), log(16, 4096)
    cap = {"f64": 8e7, "f64df": 1.6e8, "f32": 5e8, "f16": 5e8}[prec]
    steps = max(2, min(log(20, 300), int(cap / (nx * ny))))
    case = _case(kind, nx, ny, steps, prec, model, theta, nu, flow, U)
    if rng.random() < 0.5:
        case["diag"] = rng.choice([1, 10, 50])
    if rng.random() < 0.2:
        case["walls"] = True
    return case


# ----------------------------------------------------------------------------- inputs

def _fields(case, seed, nx=None, ny=None, u0=None, theta=None):
    """Initial (rho, u_x, u_y) on the GPU, (ny, nx) FP64: the flows of the benchmarks, shifted by phases
    drawn from the seed."""
    nx, ny = nx or case["nx"], ny or case["ny"]
    theta = theta or case["theta"]
    g = np.random.default_rng(seed)
    x = torch.arange(nx, dtype=torch.float64, device="cuda")[None, :]
    y = torch.arange(ny, dtype=torch.float64, device="cuda")[:, None]
    kx, ky = 2 * math.pi / nx, 2 * math.pi / ny
    one = torch.ones((ny, nx), dtype=torch.float64, device="cuda")
    U, flow = case["U"], case["flow"]
    p, q = g.uniform(0.0, 2 * math.pi, 2)
    if flow == "shocktube":
        left, right = 1.5 + 0.02 * math.sin(p), 0.75 + 0.01 * math.sin(q)
        # at rest along the tube, with a weak transverse flow that the waves carry along
        return torch.where(x < nx // 2, left, right) * one, 0.0 * one, 0.01 * torch.sin(kx * x + p) * one
    if flow == "taylor_green":
        u = u0 if u0 is not None else 0.05
        ux = -u * torch.cos(kx * x + p) * torch.sin(ky * y + q)
        uy = u * torch.sin(kx * x + p) * torch.cos(ky * y + q)
        return 1.0 - u * u / (4 * theta) * (torch.cos(2 * (kx * x + p)) + torch.cos(2 * (ky * y + q))), ux + U, uy
    if flow == "shear_wave":
        return one, U * one, 0.01 * torch.sin(kx * x + p) * one
    if flow == "shear_layer":
        width = max(2.0, ny / 50.0)
        ux = U * torch.where(y <= ny / 2, torch.tanh((y - ny / 4) / width), torch.tanh((3 * ny / 4 - y) / width))
        return one, ux * one, 0.05 * U * torch.sin(kx * x + p) * one
    # vortex: a background flow and a handful of random divergence-free modes
    ux, uy = U * one, 0.5 * U * one
    for _ in range(4):
        m, n = int(g.integers(1, 5)), int(g.integers(1, 5))
        a, p, q = 0.02 * g.uniform(0.3, 1.0), *g.uniform(0.0, 2 * math.pi, 2)
        ux = ux - a * n / max(m, n) * torch.cos(m * kx * x + p) * torch.sin(n * ky * y + q)
        uy = uy + a * m / max(m, n) * torch.sin(m * kx * x + p) * torch.cos(n * ky * y + q)
    return one, ux, uy


def _domains(case, seed):
    """(n, theta, tau, u0) of each domain: the batch benchmark's recipe, the sizes fixed by the case and the
    rest drawn from the seed."""
    sizes = [d.n for d in flows.batch_domains(case["count"], nmin=case["nx"], nmax=case["ny"])]
    ds = flows.batch_domains(case["count"], seed=seed)
    return [(n, d.theta, tau_from_nu(d.nu, d.theta), d.u0) for n, d in zip(sizes, ds)]


def _mask(case):
    mask = np.zeros((case["ny"], case["nx"]), dtype=np.uint8)
    mask[:, 0] = mask[:, -1] = 1
    return mask


# ----------------------------------------------------------------------------- the cases

def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "batch":
        ds = _domains(case, seed)
        s["fields"] = list(zip(*[_fields(case, seed + k, n, n, u0, theta) for k, (n, theta, _, u0) in enumerate(ds)]))
        n, theta, tau, _ = zip(*ds)
        s["batch"] = Batch(n, n, theta, tau, case["model"], case["prec"])
        return s
    s["fields"] = _fields(case, seed)
    s["lattice"] = lat = Lattice(case["nx"], case["ny"], case["theta"], tau_from_nu(case["nu"], case["theta"]),
                                 case["model"], case["prec"])
    if case.get("diag"):
        lat.set_diagnostics_interval(case["diag"])
    if case.get("walls"):
        lat.set_walls(_mask(case))
    if case["kind"] == "grad":
        s["fields"] = tuple(f.clone().requires_grad_(True) for f in s["fields"])
        s["target"] = _fields(case, seed + 1)
    if case["kind"] == "host":
        s["in"] = [f.cpu().pin_memory() for f in s.pop("fields")]
        s["out"] = [torch.empty_like(f).pin_memory() for f in s["in"]]
    return s


def run(s):
    case = s["case"]
    if case["kind"] == "batch":
        s["batch"].init(*s["fields"])
        s["batch"].step(case["steps"])
        return [torch.cat([m[j].reshape(-1) for m in s["batch"].moments()]) for j in range(3)]
    lat = s["lattice"]
    if case["kind"] == "host":
        total = capi.lbm_run_host(lat.ctx, *(f.data_ptr() for f in s["in"]), case["steps"],
                                  *(f.data_ptr() for f in s["out"]), want_diag=True)
        return {"fields": s["out"], "total": np.array([total[0], total[3]])}
    if case["kind"] == "grad":
        fields = run_lattice(lat, *s["fields"], case["steps"], case["every"])
        loss = sum(((f - t) ** 2).sum() for f, t in zip(fields, s["target"]))
        return {"fields": [f.detach() for f in fields], "grads": list(torch.autograd.grad(loss, s["fields"]))}
    lat.init(*s["fields"])
    lat.step(case["steps"])
    out = {"fields": list(lat.moments())}
    if case.get("diag"):
        total = lat.step_diagnostics()[0]
        out["total"] = np.array([total[0], total[3]])  # mass and kinetic energy
    return out


def _nodes(case):
    if case["kind"] == "batch":
        return sum(n * n for n, *_ in _domains(case, 0))
    return case["nx"] * case["ny"]


def work(case):
    nodes = _nodes(case)
    # three fields in, three out; the gradient also reads the target and writes three gradients. Its reverse
    # steps take at least twice the forward step's operations.
    words, passes = (12, 3) if case["kind"] == "grad" else (6, 1)
    return {"bytes": 8 * words * nodes, "flops": OPS[case["model"]] * nodes * case["steps"] * passes}


# ----------------------------------------------------------------------------- the same in plain torch, FP64

_C = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
_OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]


def _axis(u, theta):
    """Equilibrium factors of velocity components -1, 0, 1."""
    return [0.5 * (theta + u * u - u), 1.0 - theta - u * u, 0.5 * (theta + u * u + u)]


def _equilibrium(rho, u, v, theta):
    px, py = _axis(u, theta), _axis(v, theta)
    return [rho * px[a + 1] * py[b + 1] for a, b in _C]


def _moments(f):
    rho = sum(f)
    jx, jy = (f[1] + f[5] + f[8]) - (f[3] + f[6] + f[7]), (f[2] + f[5] + f[6]) - (f[4] + f[7] + f[8])
    return rho, jx / rho, jy / rho


def _collide(f, theta, tau, model):
    rho, u, v = _moments(f)
    px, py = _axis(u, theta), _axis(v, theta)
    eq = [rho * px[a + 1] * py[b + 1] for a, b in _C]
    r = 1.0 - 1.0 / tau
    if model == "lbgk":
        return [e + r * (x - e) for x, e in zip(f, eq)]
    neq = [x - e for x, e in zip(f, eq)]
    nd = 0.5 * sum((a * a - b * b) * x for (a, b), x in zip(_C, neq) if a * a != b * b)
    nxy = neq[5] + neq[7] - neq[6] - neq[8]
    k1, k2 = nd / (2 * theta**2), nxy / theta**2
    out = []
    for (a, b), e in zip(_C, eq):
        ca, cb, p = a - u, b - v, px[a + 1] * py[b + 1]
        out.append(e + r * p * (k1 * (ca * ca - cb * cb) + k2 * ca * cb))
    if model == "oreg":
        return out
    psx, psy = k1 * u * (1 - 3 * theta - u * u), -k1 * v * (1 - 3 * theta - v * v)
    psi = [0.0] * 9
    for i in (1, 2, 3, 4):
        psi[i] = -0.5 * (_C[i][0] * psx + _C[i][1] * psy)
    if model != "partial":
        mu = [(theta - w * w) * (1 - theta - w * w) / (2 * theta**2) for w in (u, v)]
        pref = -k1 if model == "complete_neq" else -0.5 * k1 * (mu[0] + mu[1])
        t = theta * (1 - 3 * theta)
        pxx = -pref * (u * u * (u * u - 1) + t)
        pyy = pref * (v * v * (v * v - 1) + t)
        pxy = pref * u * v * (u * u - v * v)
        for i in (1, 3):
            psi[i] = psi[i] + 0.5 * pyy
        for i in (2, 4):
            psi[i] = psi[i] + 0.5 * pxx
        for i in (5, 6, 7, 8):
            psi[i] = -0.25 * (pxx + pyy + _C[i][0] * _C[i][1] * pxy)
    return [o + r * p for o, p in zip(out, psi)]


def _step(f, theta, tau, model, mask):
    post = _collide(f, theta, tau, model)
    if mask is not None:
        post = [torch.where(mask, f[_OPP[i]], post[i]) for i in range(9)]
    return [torch.roll(x, (b, a), (0, 1)) for x, (a, b) in zip(post, _C)]


def _run64(fields, theta, tau, model, steps, mask=None, diag=0):
    f, total = _equilibrium(*fields, theta), None
    for t in range(steps):
        if diag and t % diag == 0:
            rho, u, v = _moments(f)
            total = np.array([float(rho.sum()), float((0.5 * rho * (u * u + v * v)).sum())])
        f = _step(f, theta, tau, model, mask)
    return _moments(f), total


def exact(case, seed):
    tau = tau_from_nu(case["nu"], case["theta"])
    theta, model, steps = case["theta"], case["model"], case["steps"]
    if case["kind"] == "batch":
        if case["count"] * steps > 15000:
            return None
        parts = [_run64(_fields(case, seed + k, n, n, u0, th), th, ta, model, steps)[0]
                 for k, (n, th, ta, u0) in enumerate(_domains(case, seed))]
        return [torch.cat([p[j].reshape(-1) for p in parts]) for j in range(3)]
    fields = _fields(case, seed)
    if case["kind"] == "grad":
        from torch.utils.checkpoint import checkpoint

        fields = [f.clone().requires_grad_(True) for f in fields]
        f = _equilibrium(*fields, theta)
        for _ in range(steps):
            f = checkpoint(lambda *a: tuple(_step(list(a), theta, tau, model, None)), *f, use_reentrant=False)
        out = _moments(list(f))
        loss = sum(((a - b) ** 2).sum() for a, b in zip(out, _fields(case, seed + 1)))
        return {"fields": [o.detach() for o in out], "grads": list(torch.autograd.grad(loss, fields))}
    mask = torch.from_numpy(_mask(case)).cuda().bool() if case.get("walls") else None
    out, total = _run64(fields, theta, tau, model, steps, mask, case.get("diag", 0))
    if case["kind"] == "host":
        rho, u, v = out
        total = np.array([float(rho.sum()), float((0.5 * rho * (u * u + v * v)).sum())])
        return {"fields": [o.cpu() for o in out], "total": total}
    return {"fields": list(out)} | ({"total": total} if total is not None else {})
