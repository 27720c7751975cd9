"""Workloads of this package's public entry points, for timing it and comparing its results.

Each case is one job of a user's program: a handle with its fields on the GPU is ready
(``prepare``), the program advances it, differentiates it or analyses it, and takes the results
(``run``).  The kinds are those of the package: forward-Euler runs on single 2D and 3D grids
(Models A, B, C, Gray-Scott, N species, the further stencils), mass/energy time series, the
batched runner, the adjoint, the semi-implicit spectral solver, and the analysis of a resident
field.  ``listed`` has the representative sizes, ``draw`` spreads over the same ranges.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2109_02598_gb300 as pf

# Model coefficients and time steps of the repository's configurations.
COEFFS = {"ac": (1.0, 1.0), "ch": (1.0, 1.0, 1.0), "gs": (0.2, 0.1, 0.04, 0.06),
          "c": (1.0, 1.0, 1.0, 1.0, 1.0)}
DT = {"ac": 0.05, "ch": 0.01, "gs": 0.5, "c": 0.005, "rd": 0.2}
NF = {"ac": 1, "ch": 1, "gs": 2, "c": 2, "rd": 3}
# Three species, seven monomials 1, u, v, w, u v^2, u^2 w, w^3 (the benchmark's network).
RD3 = ((0.2, 0.05, 0.12),
       ((0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 2, 0), (2, 0, 1), (0, 0, 3)),
       ((0.03, -0.03, 0.0, 0.1, -1.0, 0.0, 0.0), (0.0, 0.0, -0.09, 0.0, 1.0, -0.4, 0.0),
        (0.0, 0.05, 0.0, -0.2, 0.0, 0.4, -0.3)))
# Floating-point operations per site and step (the stencils and the pointwise terms as written
# in the equations; both fields together), by model and dimension.
FLOPS = {("ac", 2): 13, ("ac", 3): 15, ("ch", 2): 20, ("ch", 3): 24, ("gs", 2): 28,
         ("gs", 3): 32, ("c", 2): 38, ("c", 3): 44, ("rd", 2): 90, ("rd", 3): 96}
STENCIL_FLOPS = {"std": 0, "iso": 24, "4th": 8, "iso27": 40}  # further operations of two fields


def listed():
    return [
        # A monitored run on the smallest grid: the 128^2 Model A configuration advanced ten
        # steps between samples of mass and free energy, with the library's default tuning (a
        # short job does not autotune). Launches, synchronisations and latency.
        {"name": "series_ac2d_128", "kind": "series", "model": "ac", "nx": 128, "ny": 128, "nz": 0,
         "every": 10, "steps": 50},
        # The Cahn-Hilliard configuration: 2048^2, the long conserved coarsening run.
        {"name": "ch2d_2048", "kind": "step", "model": "ch", "nx": 2048, "ny": 2048, "nz": 0,
         "stencil": "std", "steps": 500},
        # A 2D Gray-Scott grid of a size nobody tuned for: ragged rows, odd row count.
        {"name": "gs2d_1502x1111", "kind": "step", "model": "gs", "nx": 1502, "ny": 1111, "nz": 0,
         "stencil": "std", "steps": 200},
        # The headline configuration: 3D Gray-Scott 256^3, as many steps as one benchmark job.
        {"name": "gs3d_256", "kind": "step", "model": "gs", "nx": 256, "ny": 256, "nz": 256,
         "stencil": "std", "steps": 250},
        # 3D Gray-Scott on a box whose sides are no multiples of anything.
        {"name": "gs3d_210x179x150", "kind": "step", "model": "gs", "nx": 210, "ny": 179, "nz": 150,
         "stencil": "std", "steps": 100},
        # The eutectic Model C in 3D (two fields, one of them conserved).
        {"name": "c3d_128", "kind": "step", "model": "c", "nx": 128, "ny": 128, "nz": 128,
         "stencil": "std", "steps": 100},
        # Three coupled species in 3D.
        {"name": "rd3d_160x144x136", "kind": "step", "model": "rd", "nx": 160, "ny": 144, "nz": 136,
         "stencil": "std", "steps": 50},
        # The isotropic 27-point Laplacian, for patterns that must not see the lattice's axes.
        {"name": "gs3d_iso27_160", "kind": "step", "model": "gs", "nx": 160, "ny": 160, "nz": 160,
         "stencil": "iso27", "steps": 50},
        # A parameter scan: independent 2D Gray-Scott grids of uneven sizes in one batch.
        {"name": "batch_gs2d_64", "kind": "batch", "instances": 64, "side_lo": 64, "side_hi": 512,
         "steps": 1000},
        # A training step through the simulation: forward with checkpoints and the adjoint,
        # gradients of a final-state loss with respect to the initial fields and coefficients.
        {"name": "adjoint_gs2d_512", "kind": "adjoint", "nx": 512, "ny": 512, "steps": 400},
        # The paper's own solver on the largest grid of its timing table: Model C 512^2.
        {"name": "spectral_c2d_512", "kind": "spectral", "model": "c", "nx": 512, "ny": 512, "nz": 0,
         "steps": 100},
        # The analysis of a finished 3D run on the resident field: mass, free energy and the
        # radially averaged structure factor.
        {"name": "analysis_ac3d_256", "kind": "analysis", "model": "ac", "nx": 256, "ny": 256,
         "nz": 256, "bins": 32},
    ]


def _side(rng, lo, hi):
    """A side in [lo, hi], spread over its logarithm; two in three as it falls (odd ones among
    them), one in three a multiple of 16, as people choose grids."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(lo, min(hi, n if rng.random() < 2 / 3 else 16 * max(1, round(n / 16))))


def draw(rng):
    kind = rng.choice(["series", "step2", "step2", "step3", "step3", "step3", "rd", "stencil",
                       "batch", "adjoint", "spectral", "analysis"])
    if kind == "series":
        if rng.random() < 0.5:
            nx, ny, nz = _side(rng, 64, 768), _side(rng, 64, 768), 0
        else:
            nx, ny, nz = _side(rng, 32, 96), _side(rng, 32, 96), _side(rng, 32, 96)
        every = rng.choice([5, 10, 20])
        return {"kind": "series", "model": rng.choice(["ac", "ch", "c"]), "nx": nx, "ny": ny,
                "nz": nz, "every": every, "steps": 5 * every}
    if kind == "step2":
        model = rng.choice(["ac", "ch", "gs", "gs", "c"])
        return {"kind": "step", "model": model, "nx": _side(rng, 128, 2048),
                "ny": _side(rng, 128, 2048), "nz": 0, "stencil": "std",
                "steps": rng.choice([100, 200, 400])}
    if kind == "step3":
        model = rng.choice(["ac", "ch", "gs", "gs", "c"])
        top = 256 if model in ("ac", "gs") else 192
        return {"kind": "step", "model": model, "nx": _side(rng, 64, top), "ny": _side(rng, 64, top),
                "nz": _side(rng, 64, top), "stencil": "std", "steps": rng.choice([50, 100])}
    if kind == "rd":
        if rng.random() < 0.3:
            nx, ny, nz = _side(rng, 256, 2048), _side(rng, 256, 2048), 0
        else:
            nx, ny, nz = _side(rng, 64, 192), _side(rng, 64, 192), _side(rng, 64, 192)
        return {"kind": "step", "model": "rd", "nx": nx, "ny": ny, "nz": nz, "stencil": "std",
                "steps": rng.choice([20, 50])}
    if kind == "stencil":
        model = rng.choice(["ac", "gs", "gs"])
        if rng.random() < 0.3:
            return {"kind": "step", "model": model, "nx": _side(rng, 256, 2048),
                    "ny": _side(rng, 256, 2048), "nz": 0, "stencil": rng.choice(["iso", "4th"]),
                    "steps": 50}
        return {"kind": "step", "model": model, "nx": _side(rng, 64, 192), "ny": _side(rng, 64, 192),
                "nz": _side(rng, 64, 192), "stencil": rng.choice(["iso", "iso27", "iso27"]),
                "steps": rng.choice([20, 50])}
    if kind == "batch":
        lo = rng.choice([32, 64, 96])
        return {"kind": "batch", "instances": rng.randint(12, 64), "side_lo": lo,
                "side_hi": rng.choice([256, 384, 512]), "steps": rng.choice([400, 700, 1000])}
    if kind == "adjoint":
        return {"kind": "adjoint", "nx": _side(rng, 64, 640), "ny": _side(rng, 64, 640),
                "steps": rng.choice([100, 250, 400])}
    if kind == "spectral":
        model = rng.choice(["ac", "ch", "c"])
        if rng.random() < 0.6:  # the transforms' usual sides: powers of two and small multiples
            s = [64, 96, 128, 160, 192, 256, 320, 384, 512]
            nx, ny, nz = rng.choice(s), rng.choice(s), 0
        else:
            s = [32, 48, 64, 64, 80, 96]
            nx, ny, nz = rng.choice(s), rng.choice(s), rng.choice(s)
        return {"kind": "spectral", "model": model, "nx": nx, "ny": ny, "nz": nz,
                "steps": rng.choice([60, 80, 100])}
    model = rng.choice(["ac", "ch", "c"])
    if rng.random() < 0.5:
        nx, ny, nz = _side(rng, 256, 2048), _side(rng, 256, 2048), 0
    else:
        nx, ny, nz = _side(rng, 64, 224), _side(rng, 64, 224), _side(rng, 64, 224)
    return {"kind": "analysis", "model": model, "nx": nx, "ny": ny, "nz": nz,
            "bins": rng.choice([16, 32, 64])}


# ------------------------------------------------------------------------------ inputs

def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if case.get("nz") else (case["ny"], case["nx"])


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _uniform(shape, lo, hi, gen):
    return torch.rand(shape, generator=gen, device="cuda", dtype=torch.float32) * (hi - lo) + lo


def _gray_scott(shape, gen, n_seeds, side=8):
    """u = 1, v = 0, seeded cubes (squares) of (0.5, 0.25), 1 % multiplicative noise."""
    u = torch.ones(shape, device="cuda")
    v = torch.zeros(shape, device="cuda")
    idx = []
    for s in shape:
        o = torch.randint(0, s, (n_seeds, 1), generator=gen, device="cuda")
        idx.append((o + torch.arange(min(side, s), device="cuda")) % s)
    if len(shape) == 2:
        at = (idx[0][:, :, None], idx[1][:, None, :])
    else:
        at = (idx[0][:, :, None, None], idx[1][:, None, :, None], idx[2][:, None, None, :])
    u[at] = 0.5
    v[at] = 0.25
    u *= 1 + 0.01 * _uniform(shape, -1, 1, gen)
    v *= 1 + 0.01 * _uniform(shape, -1, 1, gen)
    return u, v


def _fields(case, seed):
    """Initial fields of a single grid, as the repository's recipes make them."""
    gen, shape, model = _gen(seed), _shape(case), case.get("model", "gs")
    if model == "gs":
        n = 20 if len(shape) == 3 else max(4, (shape[0] * shape[1]) // (128 * 128))
        return _gray_scott(shape, gen, n)
    if model == "rd":
        return tuple(_uniform(shape, 0.05, 0.9, gen) for _ in range(3))
    if model == "ch":
        x = _uniform(shape, -0.05, 0.05, gen)
        return (x - x.double().mean().float(),)
    if model == "c":
        return tuple(_uniform(shape, -0.5, 0.5, gen) for _ in range(2))
    return (_uniform(shape, -0.1, 0.1, gen),)


def _analysis_fields(case, seed):
    """Phase-separated fields: smoothed noise driven towards +-1, with a little noise left."""
    gen, shape = _gen(seed), _shape(case)
    out = []
    for _ in range(NF[case["model"]]):
        x = _uniform(shape, -1, 1, gen)
        for d in range(len(shape)):
            for s in (1, 2, 4):
                x = (x + torch.roll(x, s, d) + torch.roll(x, -s, d)) / 3
        x = torch.tanh(3 * x / x.std())
        out.append((x + 0.02 * _uniform(shape, -1, 1, gen)).contiguous())
    return tuple(out)


def _batch_specs(case, seed):
    r = np.random.RandomState(int(seed) % (1 << 31))
    lo, hi = math.log(case["side_lo"]), math.log(case["side_hi"])
    # the sizes belong to the scan, not to the seed: the same for every seed of a case
    q = np.random.RandomState(case["instances"])
    return [{"n": int(round(math.exp(q.uniform(lo, hi)))), "Du": 0.2, "Dv": 0.1,
             "F": float(np.float32(r.uniform(0.02, 0.06))),
             "k": float(np.float32(r.uniform(0.045, 0.07)))} for _ in range(case["instances"])]


def _batch_fields(specs, seed):
    gen = _gen(seed)
    return [_gray_scott((s["n"], s["n"]), gen, max(1, s["n"] * s["n"] // (128 * 128)))
            for s in specs]


def _grid(case, fields):
    model = case["model"]
    coeffs = pf.rd_coeffs(*RD3) if model == "rd" else COEFFS[model]
    g = pf.Grid(_shape(case), NF[model]).set_model(model, coeffs, DT[model])
    if case.get("stencil", "std") != "std":
        g.set_stencil(case["stencil"])
    return g.write_fields(fields)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "step":  # a production run: autotuned once, as the README's example does
        g = _grid(case, _fields(case, seed))
        g.autotune()
        return {"case": case, "g": g}
    if kind == "series":
        return {"case": case, "g": _grid(case, _fields(case, seed))}
    if kind == "analysis":
        return {"case": case, "g": _grid(case, _analysis_fields(case, seed))}
    if kind == "batch":
        specs = _batch_specs(case, seed)
        b = pf.Batch(specs, DT["gs"])
        for i, (u, v) in enumerate(_batch_fields(specs, seed)):
            b.write(i, 0, u)
            b.write(i, 1, v)
        b.autotune()
        return {"case": case, "b": b, "ns": [s["n"] for s in specs],
                "out": np.empty(2 * sum(s["n"] ** 2 for s in specs), dtype=np.float32)}
    if kind == "adjoint":
        u, v = _fields(case, seed)
        gen = _gen(seed + 7919)
        return {"case": case, "u": u.requires_grad_(True), "v": v.requires_grad_(True),
                "theta": torch.tensor(COEFFS["gs"], dtype=torch.float64, requires_grad=True),
                "wu": _uniform(_shape(case), -1, 1, gen), "wv": _uniform(_shape(case), -1, 1, gen)}
    sp = pf.Spectral(_shape(case), case["model"], COEFFS[case["model"]], DT[case["model"]])
    scale = 2.0 if case["model"] == "c" else 10.0  # the timing table's U(-1, 1)
    sp.write_fields([scale * f for f in _fields(case, seed)])
    return {"case": case, "sp": sp}


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "step":
        g = state["g"]
        g.step(case["steps"])
        return g.read_fields(device=True)
    if kind == "series":
        g = state["g"]
        series = g.run_series(case["steps"], case["every"], energy=True)
        return {"series": [{"mass": r["mass"], "energy": r["energy"]} for r in series],
                "fields": g.read_fields(device=True)}
    if kind == "analysis":
        g = state["g"]
        centres, mean, counts = g.structure_factor(0, case["bins"])
        return {"mass": [g.mass(f) for f in range(NF[case["model"]])], "energy": g.energy(),
                "centres": centres, "S": mean, "counts": counts}
    if kind == "batch":
        b, out, at = state["b"], state["out"], 0
        b.run(case["steps"])
        for i, n in enumerate(state["ns"]):
            for f in (0, 1):
                b.read(i, f, out=out[at:at + n * n].reshape(n, n))
                at += n * n
        return out
    if kind == "adjoint":
        u, v, theta = state["u"], state["v"], state["theta"]
        un, vn = pf.GrayScottAdjoint.apply(u, v, theta, case["steps"], DT["gs"])
        gu, gv, gt = torch.autograd.grad((un, vn), (u, v, theta), (state["wu"], state["wv"]))
        return {"u": un.detach(), "v": vn.detach(), "gu": gu, "gv": gv, "gtheta": gt}
    sp = state["sp"]
    sp.step(case["steps"])
    return sp.read_fields(device=True)


def work(case):
    kind = case["kind"]
    if kind == "batch":
        sites = sum(s["n"] ** 2 for s in _batch_specs(case, 0))
        return {"bytes": 16.0 * sites, "flops": float(sites) * case["steps"] * FLOPS["gs", 2]}
    sites = math.prod(_shape(case))
    dim = len(_shape(case))
    if kind == "adjoint":  # forward; then its adjoint, which needs every forward state again
        return {"bytes": 40.0 * sites, "flops": float(sites) * case["steps"] * (2 * 28 + 50)}
    model = case["model"]
    if kind == "analysis":
        # one read of the fields; about ten operations per site for the energy and a real
        # transform's 2.5 log2 N for the structure factor
        return {"bytes": 4.0 * sites * NF[model],
                "flops": sites * (10.0 * NF[model] + 2.5 * math.log2(sites))}
    bytes_ = 8.0 * sites * NF[model]
    if kind == "spectral":  # two real transforms per field and step, and the pointwise parts
        per = NF[model] * (2 * 2.5 * math.log2(sites) + 10)
        return {"bytes": bytes_, "flops": sites * per * case["steps"]}
    per = FLOPS[model, dim] + STENCIL_FLOPS[case.get("stencil", "std")] * NF[model] / 2
    return {"bytes": bytes_, "flops": float(sites) * per * case["steps"]}


# ------------------------------------------------------------- the same in 64 bits, plainly

def _sh(x, d, s):
    return torch.roll(x, s, d)


def _lap(x, stencil="std"):
    """Periodic Laplacian, unit spacing."""
    dims = range(x.dim())
    if stencil == "4th":
        return sum(16 * (_sh(x, d, 1) + _sh(x, d, -1)) - (_sh(x, d, 2) + _sh(x, d, -2)) - 30 * x
                   for d in dims) / 12
    faces = sum(_sh(x, d, 1) + _sh(x, d, -1) for d in dims)
    if stencil == "std":
        return faces - 2 * x.dim() * x

    def pair(y, d):
        return _sh(y, d, 1) + _sh(y, d, -1)

    edges = sum(pair(pair(x, a), b) for a in dims for b in dims if a < b)
    if stencil == "iso27":
        corners = pair(pair(pair(x, 0), 1), 2)
        return (14 * faces + 3 * edges + corners - 128 * x) / 30
    if x.dim() == 2:
        return (4 * faces + edges - 20 * x) / 6
    return (2 * faces + edges - 24 * x) / 6


def _rhs(model, f, c, stencil="std"):
    if model == "gs":
        u, v = f
        uvv = u * v * v
        return (c[0] * _lap(u, stencil) - uvv + c[2] * (1 - u),
                c[1] * _lap(v, stencil) + uvv - (c[2] + c[3]) * v)
    if model == "ac":
        return (_lap(f[0], stencil) + c[0] * f[0] - c[1] * f[0] ** 3,)
    if model == "ch":
        return (c[2] * _lap(c[1] * f[0] ** 3 - c[0] * f[0] - _lap(f[0], stencil), stencil),)
    if model == "c":
        p, m = f
        mu = c[3] * m ** 3 - c[2] * m - c[4] * p * p - _lap(m, stencil)
        return (_lap(p, stencil) + c[0] * p - c[1] * p ** 3 + 2 * c[4] * p * m, _lap(mu, stencil))
    D, E, K = RD3
    mono = []
    for e in E:
        t = torch.ones_like(f[0])
        for x, k in zip(f, e):
            t = t * x ** k
        mono.append(t)
    return tuple(D[i] * _lap(f[i]) + sum(K[i][m] * mono[m] for m in range(len(E)) if K[i][m])
                 for i in range(3))


def _euler(model, f, c, dt, n, stencil="std"):
    for _ in range(n):
        f = tuple(x + dt * r for x, r in zip(f, _rhs(model, f, c, stencil)))
    return f


def _energy(model, f, c):
    def grad2(x):
        return sum((_sh(x, d, -1) - x) ** 2 for d in range(x.dim()))

    p = f[0]
    e = 0.5 * grad2(p) - 0.5 * c[0] * p ** 2 + 0.25 * c[1] * p ** 4
    if model == "c":
        m = f[1]
        e = e + 0.5 * grad2(m) - 0.5 * c[2] * m ** 2 + 0.25 * c[3] * m ** 4 - c[4] * p * p * m
    return float(e.sum())


def _structure_factor(psi, bins):
    """Bin centres and means of S = |rho_hat|^2 / N over the full spectrum, rho = [psi > 0]."""
    shape, dim = psi.shape, psi.dim()
    s = torch.fft.fftn((psi > 0).double()).abs() ** 2 / psi.numel()
    k2 = torch.zeros(shape, dtype=torch.float64, device=psi.device)
    for d, n in enumerate(shape):
        k = 2 * math.pi * torch.fft.fftfreq(n, dtype=torch.float64, device=psi.device)
        k2 = k2 + (k ** 2).reshape([-1 if e == d else 1 for e in range(dim)])
    kmax = math.pi * math.sqrt(dim)
    b = torch.clamp((k2.sqrt() / kmax * bins).long(), max=bins - 1).reshape(-1)[1:]
    total = torch.zeros(bins, dtype=torch.float64, device=psi.device).index_add_(
        0, b, s.reshape(-1)[1:])
    count = torch.bincount(b, minlength=bins)
    centres = (torch.arange(bins, dtype=torch.float64) + 0.5) * kmax / bins
    return centres, total / count.clamp(min=1)


def _spectral(model, f, c, dt, n):
    shape = f[0].shape
    k2 = 0
    for d, s in enumerate(shape):
        fr = torch.fft.rfftfreq if d == len(shape) - 1 else torch.fft.fftfreq
        k = 2 * math.pi * fr(s, dtype=torch.float64, device=f[0].device)
        k2 = k2 + (k ** 2).reshape([-1 if e == d else 1 for e in range(len(shape))])
    if model == "ac":
        lin, non = [-k2 + c[0]], [torch.ones_like(k2)]
    elif model == "ch":
        lin, non = [c[2] * (-k2 ** 2 + c[0] * k2)], [-c[2] * k2]
    else:
        lin, non = [-k2 + c[0], -k2 ** 2 + c[2] * k2], [torch.ones_like(k2), -k2]
    A = [torch.exp(x * dt) for x in lin]
    B = [torch.where(x == 0, torch.full_like(x, dt), torch.expm1(x * dt) / torch.where(
        x == 0, torch.ones_like(x), x)) * q for x, q in zip(lin, non)]
    dims = tuple(range(len(shape)))
    h = [torch.fft.rfftn(x) for x in f]
    for _ in range(n):
        x = [torch.fft.irfftn(y, s=shape, dim=dims) for y in h]
        if model == "ac":
            nl = [-c[1] * x[0] ** 3]
        elif model == "ch":
            nl = [c[1] * x[0] ** 3]
        else:
            nl = [-c[1] * x[0] ** 3 + 2 * c[4] * x[0] * x[1], c[3] * x[1] ** 3 - c[4] * x[0] ** 2]
        h = [a * y + b * torch.fft.rfftn(z) for a, y, b, z in zip(A, h, B, nl)]
    return tuple(torch.fft.irfftn(y, s=shape, dim=dims) for y in h)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        specs = _batch_specs(case, seed)
        out = []
        for s, f in zip(specs, _batch_fields(specs, seed)):
            c = (s["Du"], s["Dv"], s["F"], s["k"])
            f = _euler("gs", tuple(x.double() for x in f), c, DT["gs"], case["steps"])
            out += [x.reshape(-1) for x in f]
        return torch.cat(out)
    if kind == "adjoint":
        u, v = (x.double().requires_grad_(True) for x in _fields(case, seed))
        th = torch.tensor(COEFFS["gs"], dtype=torch.float64, requires_grad=True)
        gen = _gen(seed + 7919)
        wu, wv = (_uniform(_shape(case), -1, 1, gen).double() for _ in range(2))
        c = th.to("cuda")
        un, vn = _euler("gs", (u, v), c, DT["gs"], case["steps"])
        gu, gv, gt = torch.autograd.grad((un, vn), (u, v, th), (wu, wv))
        return {"u": un.detach(), "v": vn.detach(), "gu": gu, "gv": gv, "gtheta": gt}
    model = case["model"]
    if kind == "analysis":
        f = tuple(x.double() for x in _analysis_fields(case, seed))
        centres, mean = _structure_factor(f[0], case["bins"])
        return {"mass": [float(x.sum()) for x in f], "energy": _energy(model, f, COEFFS[model]),
                "centres": centres, "S": mean, "counts": None}
    f = tuple(x.double() for x in _fields(case, seed))
    if kind == "spectral":
        scale = 2.0 if model == "c" else 10.0
        f = tuple((scale * x).double() for x in _fields(case, seed))
        return _spectral(model, f, COEFFS[model], DT[model], case["steps"])
    c = COEFFS.get(model)
    if kind == "series":
        series = []
        for s in range(0, case["steps"] + 1, case["every"]):
            # Model B's fields have mean zero: their mass is rounding alone, with no value here
            mass = None if model == "ch" else [float(x.sum()) for x in f]
            series.append({"mass": mass, "energy": _energy(model, f, c)})
            if s < case["steps"]:
                f = _euler(model, f, c, DT[model], case["every"])
        return {"series": series, "fields": f}
    return _euler(model, f, c, DT[model], case["steps"], case.get("stencil", "std"))
