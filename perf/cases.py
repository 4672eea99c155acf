"""The work a user has this library do, as timed cases.

A case is one call (the transform case: a forward and an inverse call) through
the public binding, on inputs made on the GPU from a seed. Iterative solves run
a fixed number of iterations (tolerance 0), as the benchmark does, so a pass is
the same work for every build. `exact` restates each call in FP64 with plain
torch (the method as in Section 3 of the paper, in the order of the CPU oracle).

Grids have axes of 8 to 512 voxels (powers of two, or one plane), media are
Boolean sphere packs or a thresholded Gaussian random field.
"""
from __future__ import annotations

import math

import torch

from paper_2312_15554_gb300 import acm

DEV = "cuda:0"
EXACT, CENTRAL = 0, 1


# ----------------------------------------------------------------------------
# the cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # the bare transform pair on a small field, as a spectral filter of a user's own calls it: latency
        {"name": "fft_64_f32", "kind": "fft", "n0": 64, "n1": 64, "n2": 64, "fp64": False, "fields": 1},
        # the paper's own experiments: a two-dimensional cell at its resolution, one load; all launches and latency
        {"name": "stokes_plane_128_f32", "kind": "stokes", "n0": 1, "n1": 128, "n2": 128, "fp64": False, "iters": 200,
         "deriv": CENTRAL, "adaptive": True, "warm": False, "porosity": 0.6, "radius": 8.0},
        # the validation cell: FP64, fixed penalties, one load, every output
        {"name": "stokes_32_f64", "kind": "stokes", "n0": 32, "n1": 32, "n2": 32, "fp64": True, "iters": 100,
         "deriv": CENTRAL, "adaptive": False, "warm": False, "porosity": 0.6, "radius": 5.0},
        # an evolving or learned start: one load from a previous velocity and multiplier, library defaults
        {"name": "stokes_64_f32_warm", "kind": "stokes", "n0": 64, "n1": 64, "n2": 64, "fp64": False, "iters": 100,
         "deriv": EXACT, "adaptive": True, "warm": True, "porosity": 0.45, "radius": 6.0},
        # the benchmark's Stokes half: three loads on the 256^3 pack, tuned tiles, adaptive penalties
        {"name": "stokes_tensor_256_f32", "kind": "stokes_tensor", "n0": 256, "n1": 256, "n2": 256, "fp64": False,
         "iters": 20, "deriv": EXACT, "adaptive": True, "fields": True, "tuned": True, "porosity": 0.35, "radius": 8.0},
        # the largest single cell: a 512^3 random field, permeability only
        {"name": "stokes_tensor_512_f32", "kind": "stokes_tensor", "n0": 512, "n1": 512, "n2": 512, "fp64": False,
         "iters": 8, "deriv": EXACT, "adaptive": True, "fields": False, "tuned": True, "porosity": 0.3, "radius": 0.0},
        # dispersion in a non-cubic cell in FP64 with the exact symbols, corrector and gradient returned
        {"name": "solute_32x64x128_f64", "kind": "solute", "n0": 32, "n1": 64, "n2": 128, "fp64": True, "iters": 50,
         "deriv": EXACT, "Pe": 10.0, "porosity": 0.5, "radius": 6.0},
        # one composition load on an ordinary cell, untuned, library defaults
        {"name": "solute_128_f32", "kind": "solute", "n0": 128, "n1": 128, "n2": 128, "fp64": False, "iters": 60,
         "deriv": CENTRAL, "Pe": 1.0, "porosity": 0.5, "radius": 8.0},
        # the benchmark's solute half: three composition loads on the 256^3 pack, tuned tiles
        {"name": "solute_tensor_256_f32", "kind": "solute_tensor", "n0": 256, "n1": 256, "n2": 256, "fp64": False,
         "iters": 20, "deriv": CENTRAL, "Pe": 10.0, "tuned": True, "porosity": 0.35, "radius": 8.0},
        # the batched recipe: half the cells at 64^3, half at 128^3, three loads each, fixed pore-scale penalties
        {"name": "batch_12_cells_f32", "kind": "batch", "cells": 12, "small": 64, "large": 128, "fp64": False,
         "iters": 20, "deriv": CENTRAL, "adaptive": False, "warm": False, "tuned": True},
        # learned warm start: inference for the three loads of four cells
        {"name": "fno_warm_start_64", "kind": "fno_warm", "n": 64, "width": 32, "modes": 12, "layers": 4, "batch": 4},
        # learned warm start: loss and gradient of one training batch at the trained size
        {"name": "fno_gradient_64", "kind": "fno_grad", "n0": 64, "n1": 64, "n2": 64, "width": 32, "modes": 12,
         "layers": 4, "batch": 4},
    ]


def _pow2(rng, lo, hi):
    return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def _shape(rng, cap):
    """Three axes of 16 to 256 with at most `cap` voxels; one in eight a plane."""
    while True:
        n = [_pow2(rng, 16, 256) for _ in range(3)]
        if rng.random() < 0.125:
            n = [1, _pow2(rng, 32, 256), _pow2(rng, 32, 256)]
        if n[0] * n[1] * n[2] <= cap:
            return {"n0": n[0], "n1": n[1], "n2": n[2]}


def _medium(rng, c):
    ax = min(n for n in (c["n0"], c["n1"], c["n2"]) if n > 1)
    return {"porosity": round(rng.uniform(0.3, 0.7), 3), "radius": round(rng.uniform(2.5, min(10.0, ax / 4.0)), 2)}


def draw(rng):
    """One more case of the ranges the listed ones stand for."""
    kind = rng.choice(["fft", "stokes", "stokes", "stokes_tensor", "stokes_tensor", "solute", "solute",
                       "solute_tensor", "batch", "fno_warm", "fno_grad"])
    fp64 = rng.random() < 0.3
    cap = (1 << 21) if fp64 else (1 << 24)
    iters = rng.randint(10, 60)
    c = {"kind": kind}
    if kind == "fft":
        while True:
            c.update(_shape(rng, cap))
            if c["n0"] > 1:
                break
        c.update(fp64=fp64, fields=rng.randint(1, 4))
    elif kind == "stokes":
        c.update(_shape(rng, cap), fp64=fp64, iters=iters, deriv=rng.randint(0, 1), adaptive=rng.random() < 0.5,
                 warm=rng.random() < 0.4)
        c.update(_medium(rng, c))
    elif kind == "stokes_tensor":
        c.update(_shape(rng, cap), fp64=fp64, iters=iters, deriv=rng.randint(0, 1), adaptive=rng.random() < 0.5,
                 fields=rng.random() < 0.7, tuned=rng.random() < 0.5)
        c.update(_medium(rng, c))
    elif kind == "solute":
        c.update(_shape(rng, cap), fp64=fp64, iters=iters, deriv=rng.randint(0, 1),
                 Pe=round(10.0 ** rng.uniform(0.0, 1.0), 2))
        c.update(_medium(rng, c))
    elif kind == "solute_tensor":
        c.update(_shape(rng, cap), fp64=fp64, iters=iters, deriv=rng.randint(0, 1),
                 Pe=round(10.0 ** rng.uniform(0.0, 1.0), 2), tuned=rng.random() < 0.5)
        c.update(_medium(rng, c))
    elif kind == "batch":
        small = rng.choice([16, 32, 64])
        c.update(cells=rng.randint(3, 14), small=small, large=min(64 if fp64 else 128, small * rng.choice([1, 2, 4])),
                 fp64=fp64, iters=rng.randint(8, 24), deriv=rng.randint(0, 1), adaptive=rng.random() < 0.5,
                 warm=rng.random() < 0.4, tuned=rng.random() < 0.5)
    elif kind == "fno_warm":
        n = rng.choice([16, 32, 64])
        c.update(n=n, width=rng.choice([8, 16, 32]), modes=rng.randint(2, min(12, n // 2 - 1)),
                 layers=rng.randint(2, 4), batch=rng.randint(1, 4))
    else:
        n = [rng.choice([16, 32, 64]) for _ in range(3)]
        c.update(n0=n[0], n1=n[1], n2=n[2], width=rng.choice([8, 16, 32]), modes=rng.randint(2, min(12, min(n) // 2 - 1)),
                 layers=rng.randint(2, 4), batch=rng.randint(1, 4))
    return c


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _sphere_pack(shape, porosity, radius, gen):
    """Boolean pack: random voxels carry spheres (disks in a plane cell) of one radius; expected porosity as given."""
    n0, n1, n2 = shape
    ax = [torch.arange(n, device=DEV, dtype=torch.float64) for n in shape]
    ax = [torch.minimum(a, n - a) for a, n in zip(ax, shape)]
    ball = (ax[0][:, None, None] ** 2 + ax[1][None, :, None] ** 2 + ax[2][None, None, :] ** 2 <= radius * radius)
    p = 1.0 - porosity ** (1.0 / float(ball.sum()))
    seeds = torch.rand(shape, device=DEV, generator=gen) < p
    seeds[n0 // 2, n1 // 2, n2 // 2] = True
    cover = torch.fft.irfftn(torch.fft.rfftn(seeds.float()) * torch.fft.rfftn(ball.float()), s=shape)
    return (cover > 0.5).to(torch.uint8).contiguous()


def _random_field(shape, corr, gen):
    """Gaussian random field with Gaussian correlation length `corr` voxels, unit variance in expectation."""
    f = torch.fft.rfftn(torch.randn(shape, device=DEV, generator=gen))
    for a, n in enumerate(shape):
        m = (torch.fft.rfftfreq if a == 2 else torch.fft.fftfreq)(n, device=DEV) * 2.0 * math.pi
        w = torch.exp(-0.25 * (m * corr) ** 2)
        f *= w.reshape([-1 if i == a else 1 for i in range(3)])
    f = torch.fft.irfftn(f, s=shape)
    return f / f.std()


def _medium_of(case, gen):
    shape = (case["n0"], case["n1"], case["n2"])
    if case["radius"] > 0:
        return _sphere_pack(shape, case["porosity"], case["radius"], gen)
    f = _random_field(shape, 16.0, gen)
    z = math.sqrt(2.0) * float(torch.erfinv(torch.tensor(2.0 * case["porosity"] - 1.0, dtype=torch.float64)))
    return (f > z).to(torch.uint8).contiguous()


def _flow(H, gen):
    """A smooth random flow through the pores, largest speed 1 (the scaling of a converged velocity)."""
    u = torch.stack([0.4 * _random_field(tuple(H.shape), 3.0, gen) + (1.0 if c == 0 else 0.0) for c in range(3)])
    u = u * (H == 0)
    return (u / u.abs().max()).contiguous()


def _real(case):
    return torch.float64 if case["fp64"] else torch.float32


def _init_state(H, loads, gen, dtype):
    """A start near a solution's size: velocity ~1e-4 in the pores, multiplier on the solid."""
    u = 1e-4 * torch.randn((loads, 3) + tuple(H.shape), device=DEV, generator=gen) * (H == 0)
    lam = torch.randn((loads, 3) + tuple(H.shape), device=DEV, generator=gen) * (H != 0)
    return u.to(dtype).contiguous(), lam.to(dtype).contiguous()


def _fno_theta(width, modes, layers, gen):
    """Initial parameters with the scaling the training uses."""
    def u(n, s):
        return (2.0 * torch.rand(n, device=DEV, generator=gen) - 1.0) * s
    nm = 4 * modes ** 3
    parts = [u(width * 4, 0.5), u(width, 0.1)]
    for _ in range(layers):
        parts += [torch.rand(nm * width * width * 2, device=DEV, generator=gen) / (width * width),
                  u(width * width, width ** -0.5), u(width, 0.1)]
    parts += [u(6 * width, width ** -0.5), u(6, 0.1)]
    return torch.cat(parts).contiguous()


def _penalties(case):
    """Fixed-penalty cases give their penalties (the validation cell's 300); adaptive ones take the defaults."""
    if case["adaptive"]:
        return {"adaptive": 1}
    if case["kind"] == "batch":
        return {"adaptive": 0, "pore_scale": 9.0}
    return {"adaptive": 0, "alpha0": 300.0, "beta0": 300.0, "b0": 300.0}


def _batch_shapes(case):
    return [((case["small"],) if i % 2 == 0 else (case["large"],)) * 3 for i in range(case["cells"])]


def _batch_cells(case, gen, rnd):
    out = []
    for sh in _batch_shapes(case):
        r = 3.0 + float(torch.rand(1, generator=rnd)) * (min(10.0, sh[0] / 4.0) - 3.0)
        out.append(_sphere_pack(sh, 0.2 + 0.4 * float(torch.rand(1, generator=rnd)), r, gen))
    return out


G_LOAD = (1.0, 0.25, -0.5)
G_CHI = (1.0, 0.0, 0.5)


def _inputs(case, seed):
    """The tensors of a case (shared by prepare and exact)."""
    gen = _gen(seed)
    kind = case["kind"]
    if kind == "fft":
        shape = (case["fields"], case["n0"], case["n1"], case["n2"])
        return {"x": torch.randn(shape, device=DEV, generator=gen, dtype=torch.float64).to(_real(case))}
    if kind in ("stokes", "stokes_tensor"):
        s = {"H": _medium_of(case, gen)}
        if case.get("warm"):
            u, lam = _init_state(s["H"], 1, gen, _real(case))
            s["init_u"], s["init_lambda"] = u[0], lam[0]
        return s
    if kind in ("solute", "solute_tensor"):
        H = _medium_of(case, gen)
        return {"H": H, "u": _flow(H, gen).to(_real(case)).contiguous()}
    if kind == "batch":
        rnd = torch.Generator()
        rnd.manual_seed(int(seed))
        s = {"H": _batch_cells(case, gen, rnd)}
        if case["warm"]:
            st = [_init_state(h, 3, gen, _real(case)) for h in s["H"]]
            s["init_u"], s["init_lambda"] = [a for a, _ in st], [b for _, b in st]
        return s
    shape = (case["n"],) * 3 if kind == "fno_warm" else (case["n0"], case["n1"], case["n2"])
    s = {"theta": _fno_theta(case["width"], case["modes"], case["layers"], gen)}
    r = max(2.5, min(shape) / 12.0)
    s["H"] = torch.stack([_sphere_pack(shape, 0.3 + 0.1 * b, r, gen) for b in range(case["batch"])])
    if kind == "fno_grad":
        s["target"] = torch.stack([torch.stack([_random_field(shape, 2.0, gen) for _ in range(6)])
                                   for _ in range(case["batch"])])
    return s


def prepare(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    s["case"] = case
    if kind in ("fno_warm", "fno_grad"):
        shape = tuple(s["H"].shape[1:])
        s["net"] = acm.acm_fno(shape, case["width"], case["modes"], case["layers"], max_batch=case["batch"])
        s["net"].set_params(s["theta"])
        if kind == "fno_warm":
            s["init_u"] = torch.zeros((case["batch"], 3, 3) + shape, device=DEV)
            s["init_lambda"] = torch.zeros_like(s["init_u"])
        else:
            s["grad"] = torch.zeros(s["net"].num_params, device=DEV)
        return s
    dt = _real(case)
    pr = acm.FP64 if case["fp64"] else acm.FP32
    if kind == "batch":
        s["batch"] = acm.acm_batch(_batch_shapes(case))
        if case["tuned"]:
            acm.acm_batch_autotune(s["batch"], case["fp64"], case["deriv"])
        s["params"] = acm.stokes_params(eps=0.0, max_iter=case["iters"], precision=pr, deriv=case["deriv"],
                                        **_penalties(case))
        s["out"] = [torch.zeros((3, 3) + sh, dtype=dt, device=DEV) for sh in _batch_shapes(case)]
        return s
    shape = (case["n0"], case["n1"], case["n2"])
    s["ctx"] = acm.acm_ctx(shape)
    if case.get("tuned"):
        acm.acm_autotune(s["ctx"], case["fp64"], case["deriv"])
    if kind == "fft":
        s["spec"] = torch.zeros((case["fields"],) + shape[:2] + (shape[2] // 2 + 1, 2), dtype=dt, device=DEV)
        s["back"] = torch.zeros((case["fields"],) + shape, dtype=dt, device=DEV)
    elif kind in ("stokes", "stokes_tensor"):
        s["params"] = acm.stokes_params(eps=0.0, max_iter=case["iters"], precision=pr, deriv=case["deriv"],
                                        **_penalties(case))
        if kind == "stokes":
            s["u"] = torch.zeros((3,) + shape, dtype=dt, device=DEV)
            s["p"] = torch.zeros(shape, dtype=dt, device=DEV)
            s["lam"] = torch.zeros((3,) + shape, dtype=dt, device=DEV)
        elif case["fields"]:
            s["u3"] = torch.zeros((3, 3) + shape, dtype=dt, device=DEV)
    else:
        s["params"] = acm.advdiff_params(eps=0.0, max_iter=case["iters"], precision=pr, deriv=case["deriv"])
        if kind == "solute":
            s["chi"] = torch.zeros(shape, dtype=dt, device=DEV)
            s["grad"] = torch.zeros((3,) + shape, dtype=dt, device=DEV)
        else:
            s["chi"] = torch.zeros((3,) + shape, dtype=dt, device=DEV)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "fft":
        acm.acm_fft_r2c(s["ctx"], s["x"], s["spec"], case["fp64"], case["fields"])
        acm.acm_fft_c2r(s["ctx"], s["spec"], s["back"], case["fp64"], case["fields"])
        return {"spec": s["spec"], "back": s["back"]}
    if kind == "stokes":
        _, K, rep = acm.acm_stokes(s["ctx"], s["H"], G_LOAD, s["params"], s.get("init_u"), s.get("init_lambda"),
                                   s["u"], s["p"], s["lam"])
        return {"u": s["u"], "p": s["p"], "lam": s["lam"], "K": K, "iters": rep.iters}
    if kind == "stokes_tensor":
        _, K, _, reps = acm.acm_stokes_tensor(s["ctx"], s["H"], s["params"], s.get("u3"))
        out = {"K": K, "iters": [r.iters for r in reps]}
        if case["fields"]:
            out["u"] = [s["u3"][j] for j in range(3)]
        return out
    if kind == "solute":
        _, D, Dx, rep = acm.acm_advdiff(s["ctx"], s["H"], s["u"], case["Pe"], G_CHI, s["params"], s["chi"], s["grad"])
        return {"chi": s["chi"], "grad": s["grad"], "D": D, "Dx": Dx, "iters": rep.iters}
    if kind == "solute_tensor":
        _, D, Dx, reps = acm.acm_advdiff_tensor(s["ctx"], s["H"], s["u"], case["Pe"], s["params"], s["chi"])
        return {"chi": s["chi"], "D": D, "Dx": Dx, "iters": [r.iters for r in reps]}
    if kind == "batch":
        _, K, reps = acm.acm_batch_stokes(s["batch"], s["H"], s["params"], u_out=s["out"], init_u=s.get("init_u"),
                                          init_lambda=s.get("init_lambda"))
        return {"K": K, "u": s["out"], "iters": [r.iters for rs in reps for r in rs]}
    if kind == "fno_warm":
        s["net"].warm_start(s["H"], s["init_u"], s["init_lambda"])
        return {"u": s["init_u"], "lam": s["init_lambda"]}
    loss = s["net"].backward(s["H"], s["target"], s["grad"])
    return {"loss": loss, "grad": s["grad"]}


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def _stokes_work(shape, loads, iters, es, solid, fields):
    """Per iteration and load the state is read and written once (velocity, multiplier on the solid, pressure);
    six real transforms and about 60 operations a voxel."""
    V = shape[0] * shape[1] * shape[2]
    state = V * es * (3.0 + 3.0 * solid + 1.0)
    lg = math.log2(V)
    return (V + loads * (2.0 * iters * state + fields * V * es), loads * iters * V * (6 * 2.5 * lg + 60.0))


def work(case):
    kind = case["kind"]
    if kind in ("fno_warm", "fno_grad"):
        n = (case["n"],) * 3 if kind == "fno_warm" else (case["n0"], case["n1"], case["n2"])
        V, W, L, M, B = n[0] * n[1] * n[2], case["width"], case["layers"], 4 * case["modes"] ** 3, case["batch"]
        fwd = B * L * (V * W * (2.0 * 2.5 * math.log2(V) + 2.0 * W) + M * 8.0 * W * W)
        params = 2.0 * L * M * W * W
        if kind == "fno_warm":
            # each layer's weights (BF16) and its activations (BF16, in and out), for each of the three loads
            return {"bytes": 3.0 * (2.0 * params + B * V * (1 + 24.0 + L * 4.0 * W)), "flops": 3.0 * fwd}
        # forward and backward: weights twice, activations and pre-activations written and read, the gradient written
        return {"bytes": 2 * 2.0 * params + 4.0 * params + B * V * (1 + 24.0 + L * 12.0 * W), "flops": 3.0 * fwd}
    es = 8 if case["fp64"] else 4
    if kind == "fft":
        n = (case["n0"], case["n1"], case["n2"])
        V = n[0] * n[1] * n[2]
        S = n[0] * n[1] * (n[2] // 2 + 1)
        return {"bytes": case["fields"] * 2.0 * (V * es + 2.0 * S * es),
                "flops": case["fields"] * 2.0 * 2.5 * V * math.log2(V)}
    if kind == "batch":
        b = f = 0.0
        for sh in _batch_shapes(case):
            x, y = _stokes_work(sh, 3, case["iters"], es, 0.6, 3 + (6 if case["warm"] else 0))
            b, f = b + x, f + y
        return {"bytes": b, "flops": f}
    shape = (case["n0"], case["n1"], case["n2"])
    V = shape[0] * shape[1] * shape[2]
    if kind in ("stokes", "stokes_tensor"):
        fields = 7 if kind == "stokes" else (3 if case["fields"] else 0)
        fields += 6 if case.get("warm") else 0
        b, f = _stokes_work(shape, 1 if kind == "stokes" else 3, case["iters"], es, 1.0 - case["porosity"], fields)
        return {"bytes": b, "flops": f}
    loads = 1 if kind == "solute" else 3
    # the corrector read and written once an iteration, the velocity (pores only) once an iteration for all loads
    b = V + case["iters"] * V * es * (2.0 * loads + 3.0 * case["porosity"]) + loads * V * es * (4 if loads == 1 else 1)
    return {"bytes": b, "flops": loads * case["iters"] * V * (6 * 2.5 * math.log2(V) + 60.0)}


# ----------------------------------------------------------------------------
# the same calls in FP64 with plain torch
# ----------------------------------------------------------------------------
def _axis_symbols(n, deriv):
    if n == 1:
        z = torch.zeros(1, dtype=torch.float64, device=DEV)
        return z, z.clone()
    m = torch.arange(n, device=DEV, dtype=torch.float64)
    m = torch.where(m < n // 2, m, m - n)
    k = 2.0 * math.pi * m
    if deriv == EXACT:
        d = k.clone()
        d[n // 2] = 0.0
        return d, k * k
    d = torch.sin(k / n) * n
    d[n // 2] = 0.0
    return d, 4.0 * torch.sin(0.5 * k / n) ** 2 * n * n


def _symbols(shape, deriv):
    """d_c (broadcastable) and L on the half spectrum, and the Parseval weights of its columns."""
    d, L = [], 0.0
    for a in range(3):
        da, la = _axis_symbols(shape[a], deriv)
        if a == 2:
            da, la = da[: shape[2] // 2 + 1], la[: shape[2] // 2 + 1]
        view = [-1 if i == a else 1 for i in range(3)]
        d.append(da.reshape(view))
        L = L + la.reshape(view)
    w = torch.full((shape[2] // 2 + 1,), 2.0, dtype=torch.float64, device=DEV)
    w[0] = w[-1] = 1.0
    return d, L, w


def _fft(x):
    return torch.fft.rfftn(x, dim=(-3, -2, -1))


def _ifft(x, shape):
    return torch.fft.irfftn(x, s=shape, dim=(-3, -2, -1))


def _exact_stokes(H, g, case, pore_scale=0.0, init_u=None, init_lambda=None):
    """Section 3.1: ADMM with a = H lambda; returns u, lambda, p and the mean of u."""
    shape = tuple(H.shape)
    V = float(H.numel())
    Hf = H.double()
    d, L, w = _symbols(shape, case["deriv"])
    dd = d[0] ** 2 + d[1] ** 2 + d[2] ** 2
    ax = [n for n in shape if n > 1]
    psi0 = (math.pi * float(torch.tensor(ax, dtype=torch.float64).prod()) ** (1.0 / len(ax))) ** 2 / 8.0
    if case["adaptive"]:
        psi = [psi0] * 3
    elif pore_scale > 0:
        faces = sum(float((H != torch.roll(H, 1, a)).sum()) for a in range(3) if shape[a] > 1)
        l = (V - float(Hf.sum())) / faces
        psi = [psi0 * pore_scale / l ** 2] * 3
    else:
        psi = [300.0] * 3
    low = [1e-3 * x for x in psi]
    u = torch.zeros((3,) + shape, dtype=torch.float64, device=DEV) if init_u is None else init_u.double()
    lam = torch.zeros_like(u) if init_lambda is None else init_lambda.double() * Hf
    ut = u.clone()
    qh = torch.zeros(shape[:2] + (shape[2] // 2 + 1,), dtype=torch.complex128, device=DEV)
    dv = torch.zeros_like(qh)
    if init_u is not None:
        uh = _fft(u)
        dv = 1j * (d[0] * uh[0] + d[1] * uh[1] + d[2] * uh[2])
    if init_lambda is not None:
        ah = _fft(lam)
        num = 1j * (d[0] * ah[0] + d[1] * ah[1] + d[2] * ah[2])
        qh = torch.where(dd > 0, num / torch.where(dd > 0, dd, torch.ones_like(dd)), torch.zeros_like(num))

    def parseval(x):
        return math.sqrt(float((w * (x.real ** 2 + x.imag ** 2)).sum()) / V)

    for _ in range(case["iters"]):
        al, be, b = psi
        r = _fft(b * ut - lam)
        for c in range(3):
            r[c] -= 1j * d[c] * qh
            r[c][0, 0, 0] += g[c] * V
        c0 = L + b
        du = (d[0] * r[0] + d[1] * r[1] + d[2] * r[2]) / (c0 + be * dd)
        for c in range(3):
            r[c] = (r[c] - be * d[c] * du) / c0
        dv_new = 1j * du
        qh = qh - be * dv_new
        un = _ifft(r, shape)
        s = b / (b + al * Hf)
        utn = s * un
        lam = lam + al * Hf * utn
        if case["adaptive"]:
            norm = torch.linalg.vector_norm
            res = [float(norm(Hf * utn)), al * float(norm(Hf * (utn - ut))), parseval(dv_new),
                   be * parseval(dv_new - dv), float(norm(un - utn)), b * float(norm(un - u))]
            for k, tau in enumerate((5.0, 10.0, 5.0)):
                rp, rd = res[2 * k], res[2 * k + 1]
                if rp > tau * rd:
                    psi[k] = 1.1 * psi[k]
                elif rd > tau * rp:
                    psi[k] = max(psi[k] / 1.1, low[k])
        u, ut, dv = un, utn, dv_new
    p = _ifft(qh, shape)
    return u, lam, p - p.mean(), u.reshape(3, -1).mean(dim=1)


def _exact_solute(H, u, Pe, g, case):
    """Section 3.2: Lippmann-Schwinger; returns chi, its gradient, D g and its extended-domain form."""
    shape = tuple(H.shape)
    Hf, u = H.double(), u.double()
    pore = H == 0
    eta, A0 = 0.01, 0.55
    d, L, _ = _symbols(shape, case["deriv"])
    A = (1.0 - Hf) + eta * Hf
    B = Pe * (1.0 - Hf) * u
    ubar = torch.stack([x[pore].mean() for x in u])
    B0 = B.reshape(3, -1).mean(dim=1)
    gv = torch.tensor(g, dtype=torch.float64, device=DEV).reshape(3, 1, 1, 1)
    F = Pe * (1.0 - Hf) * float((ubar.reshape(3, 1, 1, 1) * gv).sum())
    den = 1j * (float(B0[0]) * d[0] + float(B0[1]) * d[1] + float(B0[2]) * d[2]) + A0 * L
    den[0, 0, 0] = 1.0
    grad = torch.zeros((3,) + shape, dtype=torch.float64, device=DEV)
    for _ in range(case["iters"]):
        e = grad + gv
        sh = _fft(F - ((B - B0.reshape(3, 1, 1, 1)) * e).sum(dim=0))
        th = _fft((A - A0) * e)
        ch = (sh + 1j * (d[0] * th[0] + d[1] * th[1] + d[2] * th[2])) / den
        ch[0, 0, 0] = 0.0
        grad = _ifft(torch.stack([1j * d[c] * ch for c in range(3)]), shape)
    chi = _ifft(ch, shape)
    pe = Pe * (ubar.reshape(3, 1, 1, 1) - u) * chi * (1.0 - Hf)
    V = float(H.numel())
    D = (((gv + grad) * (1.0 - Hf) + pe).reshape(3, -1).sum(dim=1)) / V
    Dx = ((A * (gv + grad) + pe).reshape(3, -1).sum(dim=1)) / V
    return chi, grad, D, Dx


def _unit(j):
    return tuple(1.0 if c == j else 0.0 for c in range(3))


def _exact_fno(case, theta, H, target=None):
    """The network of the learned warm start in FP64 on the BF16-rounded parameters; with a target the loss and its
    gradient by autograd."""
    W, md, Ls, B = case["width"], case["modes"], case["layers"], H.shape[0]
    shape = tuple(H.shape[1:])
    V = shape[0] * shape[1] * shape[2]
    nm = 4 * md ** 3
    th = theta.to(torch.bfloat16).double().requires_grad_(target is not None)
    at = [0]

    def take(*sh):
        n = math.prod(sh)
        at[0] += n
        return th[at[0] - n: at[0]].reshape(sh)

    P, p = take(W, 4), take(W)
    layers = [(take(nm, W, W, 2), take(W, W), take(W)) for _ in range(Ls)]
    Q, q = take(6, W), take(6)
    x = [((torch.arange(n, device=DEV, dtype=torch.float64) + 0.5) / n) for n in shape]
    f = torch.stack([torch.stack([H[b].double()] + list(torch.meshgrid(*x, indexing="ij"))) for b in range(B)])
    v = torch.einsum("ca,bazyx->bczyx", P, f) + p.reshape(1, W, 1, 1, 1)
    k0, k1 = (torch.cat([torch.arange(md), torch.arange(n - md, n)]).to(DEV) for n in shape[:2])
    for R, M, m in layers:
        vh = torch.fft.rfftn(v, dim=(-3, -2, -1))
        X = vh[:, :, k0][:, :, :, k1][..., :md].reshape(B, W, nm)
        Y = torch.einsum("mij,bjm->bim", torch.view_as_complex(R.contiguous()), X).reshape(B, W, 2 * md, 2 * md, md)
        rows = torch.zeros((B, W, 2 * md, shape[1], md), dtype=torch.complex128, device=DEV).index_copy(3, k1, Y)
        full = torch.zeros((B, W, shape[0], shape[1], md), dtype=torch.complex128, device=DEV).index_copy(2, k0, rows)
        y = torch.fft.irfftn(torch.nn.functional.pad(full, (0, shape[2] // 2 + 1 - md)), s=shape, dim=(-3, -2, -1))
        z = y + torch.einsum("ij,bjzyx->bizyx", M, v) + m.reshape(1, W, 1, 1, 1)
        v = torch.nn.functional.gelu(z)
    out = torch.einsum("oc,bczyx->bozyx", Q, v) + q.reshape(1, 6, 1, 1, 1)
    if target is None:
        return out
    mask = torch.cat([torch.ones((B, 3) + shape, device=DEV, dtype=torch.float64),
                      H.double().unsqueeze(1).expand((B, 3) + shape)], dim=1)
    loss = (((out - target.double()) * mask) ** 2).sum() / (B * V)
    (grad,) = torch.autograd.grad(loss, th)
    return loss.detach(), grad


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    if kind == "fft":
        x = s["x"].double()
        return {"spec": torch.view_as_real(_fft(x)).contiguous(), "back": x}
    if kind == "stokes":
        u, lam, p, K = _exact_stokes(s["H"], G_LOAD, case, 0.0, s.get("init_u"), s.get("init_lambda"))
        return {"u": u, "p": p, "lam": lam, "K": K, "iters": None}
    if kind == "stokes_tensor":
        us, Ks = [], []
        for j in range(3):
            u, _, _, K = _exact_stokes(s["H"], _unit(j), case)
            us.append(u if case["fields"] else None)
            Ks.append(K)
        out = {"K": torch.stack(Ks, dim=1), "iters": None}
        if case["fields"]:
            out["u"] = us
        return out
    if kind == "solute":
        chi, grad, D, Dx = _exact_solute(s["H"], s["u"], case["Pe"], G_CHI, case)
        return {"chi": chi, "grad": grad, "D": D, "Dx": Dx, "iters": None}
    if kind == "solute_tensor":
        r = [_exact_solute(s["H"], s["u"], case["Pe"], _unit(j), case) for j in range(3)]
        return {"chi": torch.stack([x[0] for x in r]), "D": torch.stack([x[2] for x in r], dim=1),
                "Dx": torch.stack([x[3] for x in r], dim=1), "iters": None}
    if kind == "batch":
        Ks, us = [], []
        for i, H in enumerate(s["H"]):
            r = [_exact_stokes(H, _unit(j), case, 9.0, s["init_u"][i][j] if case["warm"] else None,
                               s["init_lambda"][i][j] if case["warm"] else None) for j in range(3)]
            Ks.append(torch.stack([x[3] for x in r], dim=1))
            us.append(torch.stack([x[0] for x in r]))
        return {"K": torch.stack(Ks), "u": us, "iters": None}
    if kind == "fno_warm":
        us, lams = [], []
        for j in range(3):
            # load e_j: the cell with axes 0 and j swapped, fields and components swapped back
            perm = [0, 1, 2]
            perm[0], perm[j] = j, 0
            Hj = s["H"].permute(0, *[1 + a for a in perm]).contiguous()
            o = torch.cat([_exact_fno(case, s["theta"], Hj[b: b + 1]) for b in range(case["batch"])])
            o = o.permute(0, 1, *[2 + a for a in perm])
            us.append(o[:, :3][:, perm])
            lams.append(o[:, 3:][:, perm])
        return {"u": torch.stack(us, dim=1).contiguous(), "lam": torch.stack(lams, dim=1).contiguous()}
    # the loss is the mean over the samples: one sample at a time
    loss, grad = 0.0, 0.0
    for b in range(case["batch"]):
        l, g = _exact_fno(case, s["theta"], s["H"][b: b + 1], s["target"][b: b + 1])
        loss, grad = loss + l / case["batch"], grad + g / case["batch"]
    return {"loss": loss, "grad": grad}
