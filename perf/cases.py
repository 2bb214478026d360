"""The work that users of this package have it do, as cases that can be timed.

Each listed case is one call (or one short loop of calls) of the public entry
points at a size that a program of the paper's kind uses: a low-resolution
sky for a sampler's start, the Nside-64 map and its gradient, a large ragged
share of a map, the FP64 paths, the gridded field and its node gradient, an
ensemble of parameter sets, and the surrogate's evaluation, projection and
training.  `draw` gives further cases of the same ranges.

The sizes are those of the package's recipes (`inputs`), tests and benchmark.
Targets, seeds and coefficients are made from the seed by plain torch, so that
they do not depend on the code that is measured.  `exact` restates each path
in 64 bits with plain torch (Eq. 2, 5-9 and the field models for the march, a
dense multiplication for the basis, matrix products and autograd for the
network).
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2410_01136_gb300 as sx
from paper_2410_01136_gb300 import inputs
from paper_2410_01136_gb300.surrogate import Surrogate

MODELS = {"wmap": inputs.MODEL_WMAP, "jf12": inputs.MODEL_JF12, "stack": inputs.MODEL_WMAP_STACK,
          "grid": inputs.MODEL_GRID}
SIGMA_K = 0.5


def listed():
    return [
        # A low-resolution realisation, as a sampler's start or a quick look
        # takes it by the thousand: one small launch, where latency counts.
        {"name": "forward_jf12_small", "kind": "forward", "model": "jf12", "nside": 16, "n_steps": 256, "n_freq": 1,
         "f64": False, "first": 0, "count": 0},
        # The Nside-64, four-frequency simulation (the package's benchmark map).
        {"name": "forward_jf12_map", "kind": "forward", "model": "jf12", "nside": 64, "n_steps": 512, "n_freq": 4,
         "f64": False, "first": 0, "count": 0},
        # A share of a large map: the paper's stacked 16-parameter field on a
        # ragged pixel range (as shard.py cuts it) with a ragged step count.
        {"name": "forward_stack_share", "kind": "forward", "model": "stack", "nside": 128, "n_steps": 1001,
         "n_freq": 1, "f64": False, "first": 1001, "count": 98303},
        # The grid-size study of Sec. 5: a field sampled on a fine grid and
        # marched in FP64, the precision of the paper's own runs.
        {"name": "forward_grid_f64", "kind": "forward", "model": "grid", "nside": 64, "n_steps": 512, "n_freq": 1,
         "f64": True, "first": 0, "count": 0, "grid": 256},
        # The FP64 Nside-16 workload through torch autograd: maps, then the
        # gradient of a scalar of them (the forward and the reverse march).
        {"name": "autograd_wmap_f64", "kind": "autograd", "model": "wmap", "nside": 16, "n_steps": 128, "n_freq": 2,
         "f64": True, "first": 0, "count": 0},
        # Map + 16-parameter chi^2 gradient at Nside 64: one step of a fit.
        {"name": "gradient_jf12_map", "kind": "gradient", "model": "jf12", "nside": 64, "n_steps": 512, "n_freq": 4,
         "f64": False, "first": 0, "count": 0},
        # Field-level optimisation (Sec. 3.3): map, chi^2 and the gradient of
        # every node of the 128 x 128 x 32 grid.
        {"name": "gradient_grid_nodes", "kind": "grid_gradient", "model": "grid", "nside": 64, "n_steps": 512,
         "n_freq": 1, "f64": False, "first": 0, "count": 0, "grid": 128},
        # An ensemble of chains of uneven resolution with new parameters, as a
        # sampler's step or a parameter scan hands it to the batch.
        {"name": "batch_ensemble", "kind": "batch", "model": "jf12", "n_sets": 48, "max_nside": 64, "max_steps": 512,
         "n_freq": 4},
        # The surrogate's coefficients and their VJP for a few dozen chains.
        {"name": "surrogate_chains", "kind": "surrogate", "n": 96, "width": 1024, "depth": 4, "nside": 64,
         "n_basis": 3072},
        # The same for a population of parameter sets (the largest chunk).
        {"name": "surrogate_population", "kind": "surrogate", "n": 16384, "width": 1024, "depth": 4, "nside": 64,
         "n_basis": 3072},
        # Projection of a chunk of I/Q/U maps onto the surrogate's basis, as
        # the training set, the judge and a user's own maps go through it.
        {"name": "project_maps", "kind": "project", "rows": 384, "nside": 64, "n_basis": 3072},
        # Optimiser steps of the surrogate on a user's own batches, and the
        # weights after them.
        {"name": "surrogate_training", "kind": "training", "batch": 512, "steps": 64, "width": 1024, "depth": 4,
         "nside": 64, "n_basis": 3072},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _odd(rng, v):
    return v | 1 if rng.random() < 0.5 else v


def _share(rng, nside):
    """The whole map, or a ragged pixel range of it."""
    npix = 12 * nside * nside
    if rng.random() < 0.5:
        return 0, 0
    count = max(1, _odd(rng, int(npix * rng.uniform(0.2, 0.9))))
    return rng.randrange(npix - count + 1), count


def draw(rng):
    kind = rng.choice(["forward", "forward", "forward_f64", "autograd", "gradient", "gradient", "grid_gradient", "batch",
                       "surrogate", "surrogate", "project", "training"])
    if kind in ("forward", "forward_f64"):
        f64 = kind == "forward_f64"
        model = rng.choice(["jf12", "wmap", "stack", "grid"])
        nside = rng.choice([8, 16, 32, 64] if f64 else [8, 16, 32, 64, 128])
        first, count = _share(rng, nside)
        c = {"kind": "forward", "model": model, "nside": nside, "n_steps": _odd(rng, _log_int(rng, 48, 512)),
             "n_freq": rng.choice([1, 2, 3, 4]) if model in ("jf12", "wmap") else 1, "f64": f64, "first": first,
             "count": count}
        if model == "grid":
            c["grid"] = 4 * _log_int(rng, 8, 64)
        return c
    if kind in ("autograd", "gradient"):
        f64 = kind == "autograd" and rng.random() < 0.5
        nside = rng.choice([8, 16] if f64 else [8, 16, 32, 64])
        first, count = _share(rng, nside)
        model = rng.choice(["jf12", "wmap", "stack"])
        return {"kind": kind, "model": model, "nside": nside,
                "n_steps": _odd(rng, _log_int(rng, 48, 128 if f64 else 512)),
                "n_freq": rng.choice([1, 2, 3, 4]) if model != "stack" else 1, "f64": f64, "first": first,
                "count": count}
    if kind == "grid_gradient":
        nside = rng.choice([8, 16, 32, 64])
        first, count = _share(rng, nside)
        return {"kind": kind, "model": "grid", "nside": nside, "n_steps": _odd(rng, _log_int(rng, 64, 512)),
                "n_freq": 1, "f64": False, "first": first, "count": count, "grid": 4 * _log_int(rng, 8, 32)}
    if kind == "batch":
        return {"kind": kind, "model": rng.choice(["jf12", "wmap"]), "n_sets": _log_int(rng, 4, 48),
                "max_nside": rng.choice([16, 32, 64]), "max_steps": rng.choice([128, 256, 512]),
                "n_freq": rng.choice([1, 2, 4])}
    if kind == "surrogate":
        return {"kind": kind, "n": _odd(rng, _log_int(rng, 8, 16000)), "width": rng.choice([256, 512, 1024]),
                "depth": rng.choice([2, 3, 4]), "nside": rng.choice([16, 32, 64]),
                "n_basis": 64 * _log_int(rng, 4, 48)}
    if kind == "project":
        return {"kind": kind, "rows": 3 * _log_int(rng, 1, 128), "nside": rng.choice([16, 32, 64]),
                "n_basis": 64 * _log_int(rng, 4, 48)}
    return {"kind": "training", "batch": 64 * _log_int(rng, 1, 8), "steps": rng.randrange(8, 65),
            "width": rng.choice([256, 512, 1024]), "depth": rng.choice([2, 3, 4]), "nside": rng.choice([16, 32, 64]),
            "n_basis": 64 * _log_int(rng, 4, 48)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _generator(seed, tag):
    return torch.Generator(device="cuda").manual_seed((int(seed) * 1009 + tag) & 0x7FFFFFFF)


def _randn(shape, seed, tag, dtype=torch.float32):
    return torch.randn(shape, generator=_generator(seed, tag), device="cuda", dtype=dtype)


def _theta(model, seed, frac=0.05):
    """The model's fiducial parameters moved by a few per cent with the seed."""
    z = inputs.normal(inputs.substream(int(seed), 17), inputs.N_THETA[MODELS[model]])
    if model == "jf12":
        fid = inputs.jf12_fiducial(2)
        th = fid + frac * inputs.jf12_scales(fid) * z
    else:
        fid = {"wmap": np.array([6.0, math.radians(11.5), 0.0157, 0.4363, 1.0, inputs.N0_EARTH, 3.0, 0.03]),
               "stack": inputs.wmap_stack_theta(), "grid": inputs.grid_theta()}[model]
        th = fid * (1.0 + frac * z)
    ip = inputs.P_INDEX[MODELS[model]]
    th[ip] = min(max(th[ip], 2.8), 3.2)
    return th


def _freqs(case):
    # the box-filling models at the paper's 2.4 GHz, the others at the survey frequencies
    return (2.4e9,) if case["model"] in ("stack", "grid") else inputs.FREQS_C2[:case["n_freq"]]


def _grid_nodes(n, seed, dtype):
    """A seeded smooth field on (n, n, n/4) nodes: 8 plane waves, 4 uG."""
    nz = max(n // 4, 2)
    g = _generator(seed, 3)
    waves = torch.randint(-3, 4, (8, 3), generator=g, device="cuda").double()
    amps = torch.randn((8, 3), generator=g, device="cuda", dtype=torch.float64) * (4.0 / math.sqrt(8.0))
    phases = torch.rand(8, generator=g, device="cuda", dtype=torch.float64) * (2 * math.pi)
    ax = [torch.arange(m, device="cuda", dtype=torch.float64) / m for m in (n, n, nz)]
    out = torch.zeros((nz, n, n, 3), device="cuda", dtype=torch.float64)
    for k in range(8):
        w = torch.cos(2 * math.pi * (waves[k, 0] * ax[0][None, None, :] + waves[k, 1] * ax[1][None, :, None]
                                     + waves[k, 2] * ax[2][:, None, None]) + phases[k])
        out += w[..., None] * amps[k]
    return out.to(dtype).contiguous()


def _problem(case, seed):
    model = case["model"]
    box = model in ("stack", "grid")
    grid = None
    if model == "grid":
        grid = _grid_nodes(case["grid"], seed, torch.float64 if case["f64"] else torch.float32)
    return inputs.Problem(nside=case["nside"], n_steps=case["n_steps"], freq_hz=_freqs(case), model_id=MODELS[model],
                          theta=_theta(model, seed), box_clip=box, f64=case["f64"],
                          obs_kpc=inputs.OBS_PAPER_KPC if box else inputs.OBS_CONFIG_KPC, pix_begin=case["first"],
                          pix_count=case["count"], grid=grid)


def _target(prob, seed, sigma):
    """A mock observation: a coarse march at other parameters, plus noise."""
    model = {v: k for k, v in MODELS.items()}[prob.model_id]
    coarse = prob.replace(n_steps=min(prob.n_steps, 48), theta=_theta(model, seed + 7919))
    with torch.no_grad():
        maps = _march(coarse, torch.as_tensor(coarse.theta, device="cuda"))
    maps = maps + sigma * _randn(maps.shape, seed, 5, torch.float64)
    return maps.to(torch.float64 if prob.f64 else torch.float32)


def _sigma(case):
    return 1e-3 if case["model"] in ("stack", "grid") else SIGMA_K


def _batch_problems(case, seed):
    """Sets of uneven Nside and step count around the fiducial parameters."""
    ns = [v for v in (8, 16, 32, 64) if v <= case["max_nside"]][-3:]
    st = [v for v in (64, 128, 256, 512) if v <= case["max_steps"]][-3:]
    probs = []
    for k in range(case["n_sets"]):
        u = inputs.splitmix64(inputs.substream(case["n_sets"], k), 2)      # the sizes are the case's, not the seed's
        probs.append(inputs.Problem(nside=ns[int(u[0] % np.uint64(len(ns)))], n_steps=st[int(u[1] % np.uint64(len(st)))],
                                    freq_hz=inputs.FREQS_C2[:case["n_freq"]], model_id=MODELS[case["model"]],
                                    theta=_theta(case["model"], seed * 4099 + k)))
    return probs


def _surrogate_weights(case, seed):
    """Weights of a network as initialised for training, U(-1, 1)/sqrt(fan-in), flat."""
    widths = (16,) + (case["width"],) * case["depth"] + (3 * case["n_basis"],)
    g = _generator(seed, 11)
    parts = []
    for k, n in zip(widths[:-1], widths[1:]):
        parts.append(((2 * torch.rand(n * k, generator=g, device="cuda") - 1) / math.sqrt(k)))
        parts.append(0.02 * torch.randn(n, generator=g, device="cuda"))
    return widths, torch.cat(parts)


def _surrogate(case, seed, rows, batch=64, steps=10000):
    lo, hi = inputs.config5_box()
    sign, brows = inputs.surrogate_basis_spec(case["nside"], case["n_basis"], seed=5)
    _, flat = _surrogate_weights(case, seed)
    sur = Surrogate(16, lo, hi, sign, brows, width=case["width"], depth=case["depth"], nside=case["nside"],
                    batch=batch, max_eval=rows, map_chunk=1, total_steps=steps, init=flat.cpu().numpy())
    mean, scale = _normalization(case, seed)
    sur.set_normalization(mean.cpu().numpy(), scale)
    return sur


def _normalization(case, seed):
    return 2.0 * _randn(3 * case["n_basis"], seed, 13), 1.75


def _surrogate_theta(n, seed, tag):
    """Parameter sets in the surrogate's input box."""
    lo, hi = (torch.as_tensor(v, device="cuda") for v in inputs.config5_box())
    u = torch.rand((n, 16), generator=_generator(seed, tag), device="cuda", dtype=torch.float64)
    return (lo + (hi - lo) * u).float()


def prepare(case, seed):
    kind = case["kind"]
    if kind == "forward":
        return {"kind": kind, "prob": _problem(case, seed)}
    if kind == "autograd":
        prob = _problem(case, seed)
        g = _randn((prob.n_freq, 3, prob.n_pix_out), seed, 5, torch.float64 if prob.f64 else torch.float32)
        return {"kind": kind, "prob": prob, "theta": torch.tensor(prob.theta), "g": g}
    if kind in ("gradient", "grid_gradient"):
        prob = _problem(case, seed)
        target = _target(prob, seed, _sigma(case))
        state = {"kind": kind, "prob": prob, "target": target, "sigma": _sigma(case), "maps": torch.empty_like(target)}
        nbytes = (sx.adjoint_workspace_bytes if kind == "gradient" else sx.adjoint_grid_workspace_bytes)(prob)
        state["workspace"] = torch.empty(max(nbytes, 1), dtype=torch.uint8, device="cuda")
        if kind == "grid_gradient":
            state["nodes"] = torch.empty_like(prob.grid)
        return state
    if kind == "batch":
        probs = _batch_problems(case, seed)
        targets = [_target(p, seed + k, SIGMA_K) for k, p in enumerate(probs)]
        thetas = np.stack([_theta(case["model"], seed * 8209 + k) for k in range(len(probs))])
        return {"kind": kind, "plan": sx.BatchPlan(probs), "targets": targets, "thetas": thetas}
    if kind == "surrogate":
        return {"kind": kind, "sur": _surrogate(case, seed, case["n"]), "theta": _surrogate_theta(case["n"], seed, 21),
                "g": _randn((case["n"], 3, case["n_basis"]), seed, 22)}
    if kind == "project":
        sign, brows = inputs.surrogate_basis_spec(case["nside"], case["n_basis"], seed=5)
        lo, hi = inputs.config5_box()
        sur = Surrogate(16, lo, hi, sign, brows, width=64, depth=1, nside=case["nside"], batch=64, max_eval=64,
                        map_chunk=128)
        return {"kind": kind, "sur": sur, "maps": _sky(case, seed)}
    sur = _surrogate(case, seed, 64, batch=case["batch"])
    theta, coeffs = _training_batches(case, seed)
    return {"kind": kind, "sur": sur, "theta": theta, "coeffs": coeffs, "steps": case["steps"]}


def _sky(case, seed):
    """I/Q/U-like maps: a bright band over the plane and smaller noise."""
    npix = 12 * case["nside"] ** 2
    x = torch.linspace(-1, 1, npix, device="cuda")
    amp = torch.rand((case["rows"], 1), generator=_generator(seed, 31), device="cuda") * 100 + 1
    return (amp * torch.exp(-8 * x * x) + _randn((case["rows"], npix), seed, 32)).contiguous()


def _training_batches(case, seed):
    """Four batches of parameters and coefficients that depend smoothly on them."""
    mean, scale = _normalization(case, seed)
    mix = _randn((16, 3 * case["n_basis"]), seed, 43) * 0.4
    lo, hi = (torch.as_tensor(v, device="cuda") for v in inputs.config5_box())
    theta = [_surrogate_theta(case["batch"], seed, 50 + k) for k in range(4)]
    coeffs = []
    for t in theta:
        x = (2 * (t.double() - lo) / (hi - lo) - 1)
        coeffs.append((mean + scale * torch.sin(x @ mix.double())).float().reshape(-1, 3, case["n_basis"]))
    return theta, coeffs


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(state):
    kind = state["kind"]
    if kind == "forward":
        return sx.forward(state["prob"])
    if kind == "autograd":
        theta = state["theta"].clone().requires_grad_(True)
        maps = sx.SynaxMaps.apply(theta, state["prob"])
        maps.backward(state["g"])
        return {"maps": maps.detach(), "grad": theta.grad}
    if kind == "gradient":
        grad, chi2 = sx.adjoint(state["prob"], target=state["target"], sigma=state["sigma"], maps_out=state["maps"],
                                workspace=state["workspace"])
        return {"grad": grad, "chi2": chi2, "maps": state["maps"]}
    if kind == "grid_gradient":
        grad, nodes, chi2 = sx.adjoint_grid(state["prob"], target=state["target"], sigma=state["sigma"],
                                            maps_out=state["maps"], grid_grad=state["nodes"],
                                            workspace=state["workspace"])
        return {"grad": grad, "chi2": chi2, "maps": state["maps"], "nodes": nodes}
    if kind == "batch":
        grads, chi2 = state["plan"].run(targets=state["targets"], sigma=SIGMA_K, thetas=state["thetas"])
        return {"grads": grads, "chi2": chi2}
    if kind == "surrogate":
        coeffs, gtheta = state["sur"](state["theta"], state["g"])
        return {"coeffs": coeffs, "gtheta": gtheta}
    if kind == "project":
        return state["sur"].project(state["maps"])
    sur, losses = state["sur"], []
    for k in range(state["steps"]):
        losses.append(sur.step(state["theta"][k % 4], state["coeffs"][k % 4]))
    return {"losses": torch.cat(losses), "params": [v for layer in sur.params() for v in layer]}


# ---------------------------------------------------------------------------
# the work that a pass cannot do without
# ---------------------------------------------------------------------------

# Arithmetic and special-function operations of one forward sample without
# and per frequency, counted by hand from Eq. 2, 5-9 and the field model.
_FIELD_OPS = {"jf12": 168 + 14, "grid": 142 + 9, "wmap": 60 + 14, "stack": 99 + 25}


def _march_work(model, n_pix, n_steps, n_freq, size, passes, node_bytes=0, extra=0):
    return {"bytes": float(3 * n_freq * n_pix * size * (2 if passes > 1 else 1) + node_bytes),
            "flops": float(n_pix * n_steps * (passes * (_FIELD_OPS[model] + 10 * n_freq) + extra))}


def work(case):
    kind = case["kind"]
    if kind in ("forward", "autograd", "gradient", "grid_gradient"):
        n_pix = case["count"] or 12 * case["nside"] ** 2 - case["first"]
        size = 8 if case["f64"] else 4
        nodes = 0
        if case["model"] == "grid":
            nodes = 3 * case["grid"] ** 2 * max(case["grid"] // 4, 2) * size * (2 if kind == "grid_gradient" else 1)
        passes = {"forward": 1, "autograd": 4, "gradient": 3, "grid_gradient": 3}[kind]
        return _march_work(case["model"], n_pix, case["n_steps"], case["n_freq"], size, passes, nodes,
                           36 if kind == "grid_gradient" else 0)
    if kind == "batch":
        ws = [_march_work(case["model"], p.npix, p.n_steps, p.n_freq, 4, 3) for p in _batch_problems(case, 0)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if kind == "project":
        npix = 12 * case["nside"] ** 2
        # a fast transform: 2 log2(Nside) additions of the Sylvester factor and 12 of the order-12 one per pixel
        return {"bytes": 4.0 * case["rows"] * (npix + case["n_basis"]),
                "flops": float(case["rows"] * npix * (2 * math.log2(case["nside"]) + 12))}
    n_out = 3 * case["n_basis"]
    weights = 16 * case["width"] + (case["depth"] - 1) * case["width"] ** 2 + case["width"] * n_out
    if kind == "surrogate":
        return {"bytes": 4.0 * case["n"] * (2 * n_out + 32) + 2.0 * weights, "flops": 4.0 * case["n"] * weights}
    # per step: three products of each layer, and the weights and their two moments read and written
    return {"bytes": float(case["steps"] * (24 * weights + 4 * case["batch"] * n_out)),
            "flops": 6.0 * case["steps"] * case["batch"] * weights}


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------

def _triads(nside, first, count):
    """HEALPix RING pixel centres (Gorski et al. 2005) and their triads."""
    n, pix = nside, torch.arange(first, first + count, device="cuda", dtype=torch.int64)
    ncap, npix = 2 * n * (n - 1), 12 * n * n
    c = torch.where(pix < ncap, pix, npix - 1 - pix)
    k = ((1 + torch.sqrt(1 + 2 * c.double())) / 2).floor().long().clamp(min=1)
    k = torch.where(2 * k * (k - 1) > c, k - 1, k)
    k = torch.where(2 * k * (k + 1) <= c, k + 1, k)
    m = c - 2 * k * (k - 1)
    j = torch.where(pix < ncap, m, 4 * k - 1 - m)
    i = n + (pix - ncap).clamp(min=0) // (4 * n)
    jb = (pix - ncap) - (i - n) * 4 * n
    polar = (pix < ncap) | (pix >= npix - ncap)
    a = k.double() ** 2 / (3.0 * n * n)                               # 1 - |z|
    zc = torch.where(pix < ncap, 1 - a, a - 1)
    zb = (4 * n - 2 * i).double() / (3 * n)
    z = torch.where(polar, zc, zb)
    cosb = torch.sqrt(torch.where(polar, a * (2 - a), (1 - zb) * (1 + zb)))
    phi = math.pi * torch.where(polar, (j.double() + 0.5) / (2 * k).double(),
                                (jb.double() + 0.5 * ((i - n + 1) % 2).double()) / (2 * n))
    s, c = torch.sin(phi), torch.cos(phi)
    return (torch.stack([cosb * c, cosb * s, z], -1), torch.stack([-s, c, torch.zeros_like(s)], -1),
            torch.stack([-z * c, -z * s, cosb], -1))


def _sech2(z):
    e = torch.exp(-2 * z.abs())
    return 4 * e / (1 + e) ** 2


def _smooth(t):
    t = t.clamp(0, 1)
    return t * t * (3 - 2 * t)


def _field(prob, th, x, y, z, grid):
    """B (three components, uG), N0 and n_e at the points, for each model."""
    rho = torch.sqrt(x * x + y * y)
    c, s = x / rho, y / rho
    o = prob.obs_kpc
    norm = math.exp(math.hypot(o[0], o[1]) / 5) * math.cosh(o[2]) ** 2
    cr = torch.exp(-rho / 5) * _sech2(z) * norm
    model = prob.model_id
    if model == inputs.MODEL_JF12:
        sz = z / torch.sqrt(z * z + 0.01)
        lz = torch.sigmoid(2 * (z.abs() - 0.4) / 0.27)
        lz_c = torch.sigmoid(-2 * (z.abs() - 0.4) / 0.27)
        pitch = math.radians(11.5)
        u = torch.remainder(4 / math.pi * (torch.atan2(y, x) - torch.log(rho / 5) / math.tan(pitch)), 8.0)
        beta = 0
        for k in range(8):
            d = torch.remainder(u - k + 4, 8.0) - 4
            beta = beta + th[k] * (_smooth(d + 0.5) - _smooth(d - 0.5))
        amp = beta * (5 / rho) * _smooth((rho - 4.75) / 0.5) * _smooth((20.25 - rho) / 0.5) * lz_c
        halo = th[8] * torch.exp(-z.abs() / th[9]) * lz * torch.sigmoid(-2 * (rho - 9.22) / 0.2) * sz
        rp = rho - z.abs() / torch.tan(th[11])
        mag = torch.where(rp > 0, th[10] * torch.exp(-rp / 4.8) * (rp / rho), torch.zeros_like(rp))
        br = amp * math.sin(pitch) + mag * sz * torch.cos(th[11])
        bp = amp * math.cos(pitch) + halo
        ne = 0.025 * torch.exp(-rho / 20 - z.abs() / th[14]) + 0.1 * torch.exp(-rho / 4 - z.abs() / th[15])
        return br * c - bp * s, br * s + bp * c, mag * torch.sin(th[11]), th[12] * cr, ne
    disc = torch.exp(-rho / 20) * _sech2(z)
    if model == inputs.MODEL_GRID:
        nz, ny, nx = grid.shape[:3]
        idx, frac = [], []
        for v, length, n in ((x, prob.box_kpc[0], nx), (y, prob.box_kpc[1], ny), (z, prob.box_kpc[2], nz)):
            w = ((v + length / 2) * ((n - 1) / length)).clamp(0, n - 1)
            i = w.detach().floor().long().clamp(max=n - 2)
            idx.append(i)
            frac.append((w - i)[..., None])
        flat, b = grid.reshape(-1, 3), 0
        for q in range(8):
            wq, at = 1.0, 0
            for k, stride in enumerate((1, nx, nx * ny)):
                bit = (q >> k) & 1
                wq = wq * (frac[k] if bit else 1 - frac[k])
                at = at + (idx[k] + bit) * stride
            b = b + wq * flat[at]
        return b[..., 0], b[..., 1], b[..., 2], th[0] * cr, th[2] * disc
    inside = (rho >= 3) & (rho <= 20)
    lnr = torch.where(inside, torch.log(rho / 8), torch.zeros_like(rho))
    th_z = torch.where(inside, torch.tanh(z), torch.zeros_like(z))
    on = inside.double()

    def swirl(b0, psi0, psi1, chi0):
        psi, chi = psi0 * on + psi1 * lnr, chi0 * th_z
        ur, up = torch.cos(psi) * torch.cos(chi), torch.sin(psi) * torch.cos(chi)
        return b0 * (ur * c - up * s), b0 * (ur * s + up * c), b0 * torch.sin(chi)

    if model == inputs.MODEL_WMAP:
        env = torch.exp(-rho / 8 - z.abs())
        bx, by, bz = swirl(th[0], th[1], th[2], th[3])
        return env * bx + th[4], env * by, env * bz, th[5] * cr, th[7] * disc
    k = [swirl(*th[4 * i:4 * i + 4]) for i in range(4)]
    return (0.6 * k[0][0] + 0.3 * k[1][0] + 0.1 * k[2][2] + 0.3 * k[3][1],
            0.6 * k[0][1] + 0.3 * k[1][2] + 0.1 * k[2][1] + 0.3 * k[3][0],
            0.6 * k[0][2] + 0.3 * k[1][1] + 0.1 * k[2][0] + 0.3 * k[3][2], th[16] * cr, th[18] * disc)


def _march_chunk(prob, th, grid, first, count):
    """Eq. 2, 5-9 for `count` pixels: brightness temperatures [F, 3, count]."""
    qe, me, cc, kb, kpc = 4.803204712570263e-10, 9.1093837015e-28, 2.99792458e10, 1.380649e-16, 3.0856775814913673e21
    n, el, eb = _triads(prob.nside, first, count)
    o = torch.as_tensor(prob.obs_kpc, device="cuda", dtype=torch.float64)
    if prob.box_clip:
        h = torch.as_tensor(prob.box_kpc, device="cuda", dtype=torch.float64) / 2
        exits = torch.where(n > 0, (h - o) / n, torch.where(n < 0, (-h - o) / n, torch.full_like(n, math.inf)))
        length = exits.amin(-1, keepdim=True)
    else:
        length = torch.full((count, 1), prob.r_max_kpc, device="cuda", dtype=torch.float64)
    dr = length / prob.n_steps
    t = (torch.arange(prob.n_steps, device="cuda", dtype=torch.float64) + 0.5) * dr
    pos = [o[k] + t * n[:, k:k + 1] for k in range(3)]
    bx, by, bz, n0, ne = _field(prob, th, *pos, grid)

    def along(v):
        return bx * v[:, 0:1] + by * v[:, 1:2] + bz * v[:, 2:3]

    a, b = along(el), along(eb)
    bp2 = a * a + b * b
    dark = bp2 <= 1e-30
    bp2 = torch.where(dark, torch.ones_like(bp2), bp2)
    p = th[inputs.P_INDEX[prob.model_id]]
    j = torch.where(dark, torch.zeros_like(bp2), n0 * torch.exp((p + 1) / 4 * torch.log(bp2)))
    f = -ne * along(n) * dr
    rm = (torch.cumsum(f, -1) - 0.5 * f) * (1e-6 * kpc * qe ** 3 / (2 * math.pi * me ** 2 * cc ** 4))
    cos2, sin2 = (a * a - b * b) / bp2, 2 * a * b / bp2
    rows = []
    for nu in prob.freq_hz:
        pre = math.sqrt(3) * qe ** 3 / (8 * math.pi * me * cc ** 2)
        ln_x = math.log(4 * math.pi * nu * me * cc / (3 * qe))
        g = torch.exp((1 - p) / 2 * ln_x + (p + 1) / 2 * math.log(1e-6) + torch.lgamma(p / 4 - 1 / 12)) * pre
        to_t = kpc * cc * cc / (2 * kb * nu * nu)
        a_i = g * 2 ** ((p + 1) / 2) / (p + 1) * torch.exp(torch.lgamma(p / 4 + 19 / 12)) * to_t
        a_p = g * 2 ** ((p - 3) / 2) * torch.exp(torch.lgamma(p / 4 + 7 / 12)) * to_t
        phase = 2 * (cc / nu) ** 2 * rm
        co, si = torch.cos(phase), torch.sin(phase)
        rows.append(torch.stack([a_i * (j * dr).sum(-1), a_p * (j * (cos2 * co - sin2 * si) * dr).sum(-1),
                                 a_p * (j * (cos2 * si + sin2 * co) * dr).sum(-1)]))
    return torch.stack(rows)


def _chunks(prob, samples=1 << 21):
    per = max(1, samples // prob.n_steps)
    for first in range(0, prob.n_pix_out, per):
        yield prob.pix_begin + first, min(per, prob.n_pix_out - first), first


def _march(prob, th):
    grid = None if prob.grid is None else prob.grid.double()
    return torch.cat([_march_chunk(prob, th, grid, first, count) for first, count, _ in _chunks(prob, 1 << 23)], -1)


def _march_gradient(prob, seeds):
    """Maps, gradient and node gradient of sum(seed * maps); seeds(maps, at) gives the seed of a chunk."""
    th = torch.tensor(prob.theta, device="cuda", dtype=torch.float64, requires_grad=True)
    grid = None if prob.grid is None else prob.grid.double().requires_grad_(True)
    maps = []
    for first, count, at in _chunks(prob):
        m = _march_chunk(prob, th, grid, first, count)
        m.backward(seeds(m.detach(), slice(at, at + count)))
        maps.append(m.detach())
    return torch.cat(maps, -1), th.grad, None if grid is None else grid.grad


def _chi2(prob, target, sigma):
    total = torch.zeros((), device="cuda", dtype=torch.float64)

    def seeds(m, at):
        d = m - target[..., at].double()
        total.add_((d * d).sum() / sigma ** 2)
        return 2 * d / sigma ** 2

    maps, grad, nodes = _march_gradient(prob, seeds)
    return maps, grad, nodes, total.reshape(1)


def _network(params, depth, x):
    for k in range(depth):
        x = torch.nn.functional.gelu(x @ params[2 * k].T + params[2 * k + 1])
    return x @ params[2 * depth].T + params[2 * depth + 1]


def _network_inputs(case, seed):
    widths, flat = _surrogate_weights(case, seed)
    flat, params, o = flat.double(), [], 0
    for k, n in zip(widths[:-1], widths[1:]):
        params += [flat[o:o + n * k].reshape(n, k), flat[o + n * k:o + n * k + n]]
        o += n * k + n
    mean, scale = _normalization(case, seed)
    return params, mean.double(), scale


def _unit_box(theta):
    lo, hi = (torch.as_tensor(v, device="cuda") for v in inputs.config5_box())
    return 2 * (theta.double() - lo) / (hi - lo) - 1


def _hadamard_rows(nside, rows):
    """Rows of H_12 (x) H_M over the pixels, as a function of a pixel slice."""
    residues = {(x * x) % 11 for x in range(1, 11)}
    h12 = torch.zeros((12, 12), dtype=torch.float64)
    for i in range(12):
        for j in range(12):
            if i == 0:
                v = 0 if j == 0 else 1
            elif j == 0:
                v = -1
            else:
                d = (j - i) % 11
                v = 0 if d == 0 else (1 if d in residues else -1)
            h12[i, j] = v + (1 if i == j else 0)
    m = nside * nside
    r = torch.as_tensor(rows.astype(np.int64), device="cuda")

    def part(pix):
        bits = (r % m)[:, None] & (pix % m)[None, :]
        for k in (16, 8, 4, 2, 1):
            bits = bits ^ (bits >> k)
        return h12.cuda()[(r // m)[:, None], (pix // m)[None, :]] * (1 - 2 * (bits & 1)).double()

    return part


def exact(case, seed):
    kind = case["kind"]
    if kind == "forward":
        prob = _problem(case, seed)
        with torch.no_grad():
            return _march(prob, torch.as_tensor(prob.theta, device="cuda"))
    if kind == "autograd":
        prob = _problem(case, seed)
        g = _randn((prob.n_freq, 3, prob.n_pix_out), seed, 5, torch.float64 if prob.f64 else torch.float32).double()
        maps, grad, _ = _march_gradient(prob, lambda m, at: g[..., at])
        return {"maps": maps, "grad": grad}
    if kind in ("gradient", "grid_gradient"):
        prob = _problem(case, seed)
        maps, grad, nodes, chi2 = _chi2(prob, _target(prob, seed, _sigma(case)), _sigma(case))
        out = {"grad": grad, "chi2": chi2, "maps": maps}
        return dict(out, nodes=nodes) if kind == "grid_gradient" else out
    if kind == "batch":
        grads, chi2 = [], []
        for k, p in enumerate(_batch_problems(case, seed)):
            target = _target(p, seed + k, SIGMA_K)
            got = _chi2(p.with_theta(_theta(case["model"], seed * 8209 + k)), target, SIGMA_K)
            grads.append(got[1])
            chi2.append(got[3])
        return {"grads": torch.stack(grads), "chi2": torch.cat(chi2)}
    if kind == "project":
        npix = 12 * case["nside"] ** 2
        sign, rows = inputs.surrogate_basis_spec(case["nside"], case["n_basis"], seed=5)
        part, x = _hadamard_rows(case["nside"], rows), _sky(case, seed).double()
        x = x * torch.as_tensor(sign.astype(np.float64), device="cuda")
        out = torch.zeros((case["rows"], case["n_basis"]), device="cuda", dtype=torch.float64)
        for p0 in range(0, npix, 4096):
            pix = torch.arange(p0, min(npix, p0 + 4096), device="cuda")
            out += x[:, pix] @ part(pix).T
        return out / math.sqrt(npix)
    params, mean, scale = _network_inputs(case, seed)
    if kind == "surrogate":
        coeffs, gtheta = [], []
        lo, hi = (torch.as_tensor(v, device="cuda") for v in inputs.config5_box())
        theta, g = _surrogate_theta(case["n"], seed, 21), _randn((case["n"], 3, case["n_basis"]), seed, 22)
        for t, gc in zip(theta.split(2048), g.split(2048)):
            x = _unit_box(t).requires_grad_(True)
            y = mean + scale * _network(params, case["depth"], x)
            y.backward(gc.double().reshape(y.shape))
            coeffs.append(y.detach().reshape(-1, 3, case["n_basis"]))
            gtheta.append(x.grad * 2 / (hi - lo))
        return {"coeffs": torch.cat(coeffs), "gtheta": torch.cat(gtheta)}
    theta, data = _training_batches(case, seed)
    params = [v.clone().requires_grad_(True) for v in params]
    m, v = [torch.zeros_like(q) for q in params], [torch.zeros_like(q) for q in params]
    losses = []
    for k in range(case["steps"]):
        y = _network(params, case["depth"], _unit_box(theta[k % 4]))
        want = (data[k % 4].double().reshape(y.shape) - mean) / scale
        loss = ((y - want) ** 2).mean()
        grads = torch.autograd.grad(loss, params)
        losses.append(loss.detach().reshape(1))
        lr = 1e-5 + 0.5 * (1e-3 - 1e-5) * (1 + math.cos(math.pi * k / 10000))
        with torch.no_grad():
            for q, g, a, b in zip(params, grads, m, v):
                a.mul_(0.9).add_(g, alpha=0.1)
                b.mul_(0.999).add_(g * g, alpha=0.001)
                q -= lr * (a / (1 - 0.9 ** (k + 1))) / (torch.sqrt(b / (1 - 0.999 ** (k + 1))) + 1e-8)
    return {"losses": torch.cat(losses), "params": [q.detach() for q in params]}
