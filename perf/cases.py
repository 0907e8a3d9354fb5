"""The work that a program gives this framework, as cases that can be timed and compared.

Each case is one call (or the few calls that belong together) through the
public entry points of ``paper_2103_04856_gb300.pfc``: energies and gradients,
descent steps and runs, batches of problems, the generator of Alg. 1 alone and
batched, the Sec. 5.2 extensions, and the analysis of a generated shape.  The
listed sizes are those of the repository's workloads (``inputs.py``, the
benchmark) and odd ones; ``draw`` gives others of the same ranges.

``exact`` restates every case in plain torch in 64 bits: the energy density of
eq. Feps on rolled fields, gradients by autograd in slabs of planes, explicit
Gaussian taps and Adam.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2103_04856_gb300 import inputs as I
from paper_2103_04856_gb300 import pfc

WILLMORE = (1.0, 0.0, 1.0, 0.0, 0.0, 0.0)          # kappa1^2 + kappa2^2
GAUSS = (0.0, 1.0, 0.0, 0.0, 0.0, 0.0)             # kappa1 kappa2
TUBE = I.smaller_first_poly_to_a(1.0, 0.2, 0.0, -0.5, 0.0)
MEMBRANE = I.smaller_first_poly_to_a(0.2, 1.0, 0.3)
PAPER = (1.0, 2.4, 9.0, 30.0, 170.0, -195.0)       # the generator's setting (Fig. cvg_1)
POLYS = {"willmore": WILLMORE, "gauss": GAUSS, "tube": TUBE, "membrane": MEMBRANE, "paper": PAPER}
TAU = 1e-3
# the scale of the Adam moments of a run in progress: four times the rms of dG/dA on
# the fields of _flow_state (the moments remember the larger gradients before)
FLOW_GRAD = 128.0
# Curvatures of a unit box with h = 0.01 are a hundred times those of a grid with
# h = 1, D = 2|M|^2 - (Tr M)^2 ten thousand times: this xi smooths its kink there as
# 1e-2 does for the descent runs below.  (At 1e-6 the flow amplifies the last bit of
# an FP32 gradient to a percent of the moments within ten iterations.)
FLOW_XI = 1.0


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # the smallest call: a gradient of a 32^3 field inside somebody's own optimiser loop,
        # where the launch, the wait and the host's part count
        {"name": "grad_32", "kind": "grad", "nx": 32, "ny": 32, "nz": 32, "poly": "willmore", "eps": 1.5, "xi": 1e-6,
         "well": 0},
        # the 32^3 FP64 descent of 100 steps (the validation of a method before it is scaled up)
        {"name": "run_fp64_32", "kind": "run", "nx": 32, "ny": 32, "nz": 32, "poly": "willmore", "eps": 1.5,
         "xi": 1e-2, "prec": "fp64", "steps": 100},
        # a PyTorch program that differentiates the energy of a ragged box by autograd: no axis a
        # multiple of a tile, rows that 16-byte loads do not fit, the +-1 double well
        {"name": "autograd_ragged", "kind": "autograd", "nx": 90, "ny": 77, "nz": 61, "poly": "tube", "eps": 1.5,
         "xi": 1e-2, "well": 1},
        # energies alone (a line search): a box of odd sizes, all six coefficients
        {"name": "energy_ragged", "kind": "energy", "nx": 201, "ny": 150, "nz": 133, "poly": "paper", "eps": 1.5,
         "xi": 1e-2, "well": 0},
        # the benchmark's four validation problems at 128^3, one projected step in one batch
        {"name": "batch_step_128x4", "kind": "batch_step", "n": 128, "count": 4, "eps": 2.0, "xi": 1e-6},
        # the tube-favouring descent at 256^3, as the step loop runs it
        {"name": "run_tube_256", "kind": "run", "nx": 256, "ny": 256, "nz": 256, "poly": "tube", "eps": 1.5,
         "xi": 1e-2, "prec": "fp32", "steps": 8},
        # the largest workload: one projected step of the membrane-favouring 512^3 field
        {"name": "step_membrane_512", "kind": "step", "nx": 512, "ny": 512, "nz": 512, "poly": "membrane", "eps": 2.0,
         "xi": 1e-6},
        # a parameter study: many problems of mixed sizes and coefficients advanced together
        {"name": "batch_run_mixed", "kind": "batch_run", "lo": 64, "hi": 128, "count": 24, "eps": 1.5, "xi": 1e-2,
         "steps": 16},
        # the paper's generator at 100^3, one shape, part of its 8000 iterations
        {"name": "flow_100", "kind": "flow", "nx": 100, "ny": 100, "nz": 100, "sigma": 2.0, "steps": 32},
        # sixteen such shapes together
        {"name": "flow_batch_100x16", "kind": "flow_batch", "nx": 100, "ny": 100, "nz": 100, "count": 16, "sigma": 2.0,
         "steps": 8},
        # Sec. 5.2: spatialised coefficients a(x) with the orientation term
        {"name": "run_field_128", "kind": "run_field", "nx": 128, "ny": 128, "nz": 128, "eps": 2.0, "xi": 1e-2,
         "steps": 8},
        # what is done with a finished shape: viability, curvatures, the curvature diagram
        {"name": "analyse_200", "kind": "analyse", "nx": 200, "ny": 200, "nz": 200, "eps": 3.0},
    ]


def _size(rng, lo, hi):
    """A size in [lo, hi], uniform in its logarithm; every third is odd."""
    n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    if rng.random() < 0.34:
        n |= 1
    return min(hi, max(lo, n))


def draw(rng):
    kind = rng.choice(("grad", "grad", "autograd", "energy", "run", "run64", "step", "step", "batch_step", "batch_run",
                       "flow", "flow_batch", "run_field", "analyse"))
    box = lambda lo, hi: {"nx": _size(rng, lo, hi), "ny": _size(rng, lo, hi), "nz": _size(rng, lo, hi)}  # noqa: E731
    eps = round(rng.uniform(1.5, 2.5), 3)
    poly = rng.choice(("willmore", "tube", "membrane"))
    if kind == "grad":
        # symmetric polynomials take the default xi; the others' gradient has a kink of width xi
        return {"kind": "grad", **box(24, 256), "poly": poly, "eps": eps, "xi": 1e-6 if poly == "willmore" else 1e-2,
                "well": rng.choice((0, 1))}
    if kind == "autograd":
        return {"kind": "autograd", **box(24, 160), "poly": poly, "eps": eps, "xi": 1e-2, "well": rng.choice((0, 1))}
    if kind == "energy":
        return {"kind": "energy", **box(32, 300), "poly": rng.choice(("willmore", "tube", "paper")), "eps": eps,
                "xi": 1e-2, "well": rng.choice((0, 1))}
    if kind == "run":
        return {"kind": "run", **box(64, 256), "poly": poly, "eps": eps, "xi": 1e-2, "prec": "fp32",
                "steps": rng.choice((3, 5, 8))}
    if kind == "run64":
        return {"kind": "run", **box(16, 48), "poly": "willmore", "eps": eps, "xi": 1e-2, "prec": "fp64",
                "steps": rng.choice((33, 64, 100))}
    if kind == "step":
        return {"kind": "step", **box(96, 500), "poly": poly, "eps": eps, "xi": 1e-6}
    if kind == "batch_step":
        return {"kind": "batch_step", "n": _size(rng, 72, 160), "count": rng.randint(2, 6), "eps": 2.0, "xi": 1e-6}
    if kind == "batch_run":
        return {"kind": "batch_run", "lo": 48, "hi": rng.choice((96, 112, 128)), "count": rng.randint(6, 24),
                "eps": eps, "xi": 1e-2, "steps": rng.choice((4, 8, 16))}
    if kind == "flow":
        return {"kind": "flow", **box(60, 132), "sigma": rng.choice((1.0, 1.5, 2.0, 2.0)), "steps": rng.choice((12, 32))}
    if kind == "flow_batch":
        b = box(56, 100)
        return {"kind": "flow_batch", **b, "count": rng.randint(2, 16), "sigma": rng.choice((1.0, 2.0, 2.0)),
                "steps": rng.choice((4, 8))}
    if kind == "run_field":
        return {"kind": "run_field", **box(48, 160), "eps": 2.0, "xi": 1e-2, "steps": rng.choice((4, 8))}
    return {"kind": "analyse", **box(64, 256), "eps": 3.0}


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


# ------------------------------------------------------------------ inputs

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _noise(shape, mean, std, g, dtype=torch.float32):
    return (mean + std * torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)).to(dtype)


def _smooth(shape, g, passes=12):
    """A smooth random periodic field of unit deviation: noise under repeated 7-point means
    (a correlation length of about 7 voxels)."""
    u = torch.randn(shape, generator=g, device="cuda", dtype=torch.float64)
    for d in (0, 1, 2):
        for _ in range(passes):
            u = (u + sum(torch.roll(u, k, d) for k in (-3, -2, -1, 1, 2, 3))) / 7.0
    return u / u.std()


def _ball(n, kind, eps, g):
    """The validation shapes at 128^3: a tanh sphere or a z-periodic cylinder, its centre anywhere."""
    c = torch.rand(3, generator=g, device="cuda", dtype=torch.float64) * n
    ax = torch.arange(n, device="cuda", dtype=torch.float64)
    d = [torch.remainder(ax - c[k] + n / 2.0, float(n)) - n / 2.0 for k in range(3)]
    r2 = d[2][None, :, None] ** 2 + d[0][None, None, :] ** 2
    if kind == "sphere":
        dist = n / 4.0 - torch.sqrt(d[1][:, None, None] ** 2 + r2)
    else:
        dist = (20.0 * n / 128.0 - torch.sqrt(r2)).expand(n, n, n)
    return (0.5 * (1.0 + torch.tanh(dist / (math.sqrt(2.0) * eps)))).float().contiguous()


def _field(case, seed):
    g = _gen(seed)
    dt = torch.float64 if case.get("prec") == "fp64" else torch.float32
    mean = 0.3 if case.get("well", 0) == 0 else -0.4
    return _noise(_shape(case), mean, 0.1 if case.get("well", 0) == 0 else 0.2, g, dt)


def _problem(case):
    return pfc.Problem.from_shape(_shape(case), eps=case["eps"], a=POLYS[case["poly"]], xi=case["xi"],
                                  well=case.get("well", 0), prec=case.get("prec", "fp32"))


def _batch_problems(case):
    """The problems of a batch: the validation pairs of shape and polynomial, or mixed sizes and coefficients."""
    if case["kind"] == "batch_step":
        pairs = [("sphere", "willmore"), ("sphere", "gauss"), ("cylinder", "willmore"), ("cylinder", "gauss")]
        return [pairs[k % 4] + (case["n"],) for k in range(case["count"])]
    rng = np.random.default_rng(2103 + case["count"])      # the study's parameters: the same for every seed
    out = []
    for _ in range(case["count"]):
        n = int(rng.choice([case["lo"], (case["lo"] + case["hi"]) // 2, case["hi"]]))
        a, b = rng.uniform(0.2, 1.0, 2)
        c = rng.uniform(-0.3, 0.3)
        d, e = rng.uniform(-0.5, 0.5, 2)
        out.append((n, I.smaller_first_poly_to_a(a, b, c, d, e), float(rng.uniform(0.15, 0.45))))
    return out


def _batch_fields(case, seed):
    g = _gen(seed)
    if case["kind"] == "batch_step":
        return [_ball(n, s, case["eps"], g) for s, _, n in _batch_problems(case)]
    return [_noise((n, n, n), vf, 0.1, g) for n, _, vf in _batch_problems(case)]


def _flow_state(case, seed, count):
    """A, m, v of flows in progress: A a gradient whose divergence makes a shape of +-1 phases
    (found with FFTs) plus a little white noise, moments of a typical gradient."""
    g = _gen(seed)
    shape = _shape(case)
    h = 0.01
    k = [2.0 * math.pi * torch.fft.fftfreq(n, device="cuda", dtype=torch.float64) for n in shape]
    s = [torch.sin(t) / h for t in k]                   # symbol of the central difference
    s2 = s[0][:, None, None] ** 2 + s[1][None, :, None] ** 2 + s[2][None, None, :] ** 2
    inv = torch.where(s2 > 1.0, 1.0 / s2.clamp(min=1.0), torch.zeros_like(s2))
    out = []
    for _ in range(count):
        f = torch.fft.fftn(torch.tanh(2.0 * (_smooth(shape, g, 6) - 0.6))) * inv
        A = torch.stack([torch.fft.ifftn(f * (-1j * s[c].reshape([-1 if d == c else 1 for d in range(3)]))).real
                         for c in (2, 1, 0)])
        A = (A + 1e-5 * torch.randn((3,) + shape, generator=g, device="cuda", dtype=torch.float64)).float()
        m = _noise((3,) + shape, 0.0, 0.3 * FLOW_GRAD, g)
        v = ((0.5 + torch.rand((3,) + shape, generator=g, device="cuda", dtype=torch.float64)) * FLOW_GRAD ** 2).float()
        out.append((A.contiguous(), m, v))
    return out


FLOW_T0 = 200          # Adam steps already taken
FLOW_M0 = -0.66


def _flow_masses(count):
    return [FLOW_M0 + 0.02 * (k % 4) for k in range(count)]


def _flow_problem(case):
    return pfc.Problem.from_shape(_shape(case), eps=0.02, a=PAPER, h=0.01, xi=FLOW_XI, well=pfc.PFC_WELL_PM1)


def _coef_field(case):
    """a(x) of Sec. 5.2: two parameter sets blended along x, periodically."""
    nx = case["nx"]
    w = 0.5 * (1.0 + torch.cos(2.0 * math.pi * torch.arange(nx, device="cuda", dtype=torch.float64) / nx))
    a0 = torch.tensor(TUBE, device="cuda", dtype=torch.float64)
    a1 = torch.tensor(MEMBRANE, device="cuda", dtype=torch.float64)
    line = a0[:, None] * w + a1[:, None] * (1.0 - w)
    return line[:, None, None, :].expand((6,) + _shape(case)).float().contiguous()


THETA = (0.6, 0.0, 0.8)
MU = 0.5


def _shape_field(case, seed):
    """A generated shape: +-1 phases of a smooth random field with a tanh profile."""
    return torch.tanh(2.0 * (_smooth(_shape(case), _gen(seed)) - 0.3)).float()


# ------------------------------------------------------------------ prepare and run

def prepare(case, seed):
    k = case["kind"]
    if k in ("grad", "autograd", "energy", "step", "run"):
        s = {"case": case, "ctx": pfc.Context(_problem(case)), "u": _field(case, seed)}
        if k in ("grad", "step", "run"):
            s["out"] = torch.empty_like(s["u"])
        if k == "autograd":
            s["u"].requires_grad_(True)
        if k == "step":
            s["scalars"] = torch.zeros(5, dtype=torch.float64, device="cuda")
        return s
    if k in ("batch_step", "batch_run"):
        us = _batch_fields(case, seed)
        if k == "batch_step":
            probs = [pfc.Problem.from_shape((n, n, n), eps=case["eps"], a=POLYS[p], xi=case["xi"])
                     for _, p, n in _batch_problems(case)]
        else:
            probs = [pfc.Problem.from_shape((n, n, n), eps=case["eps"], a=a, xi=case["xi"])
                     for n, a, _ in _batch_problems(case)]
        return {"case": case, "batch": pfc.Batch(probs), "u": us, "out": [torch.empty_like(u) for u in us]}
    if k == "flow":
        return {"case": case, "flow": pfc.HFlow(_flow_problem(case), m0=FLOW_M0, blur_sigma=case["sigma"]),
                "init": _flow_state(case, seed, 1)[0],
                "work": [torch.empty((3,) + _shape(case), device="cuda") for _ in range(3)]}
    if k == "flow_batch":
        n = case["count"]
        init = _flow_state(case, seed, n)
        return {"case": case, "init": init,
                "flow": pfc.HFlowBatch([_flow_problem(case)] * n, _flow_masses(n), blur_sigma=case["sigma"]),
                "work": [[torch.empty_like(x) for x in t] for t in init]}
    if k == "run_field":
        prob = pfc.Problem.from_shape(_shape(case), eps=case["eps"], a=TUBE, xi=case["xi"], mu=MU, theta=THETA)
        ctx = pfc.Context(prob)
        ctx.set_coefficient_field(_coef_field(case))
        u = _noise(_shape(case), 0.3, 0.1, _gen(seed))
        return {"case": case, "ctx": ctx, "u": u, "out": torch.empty_like(u)}
    prob = pfc.Problem.from_shape(_shape(case), eps=case["eps"], a=WILLMORE, well=pfc.PFC_WELL_PM1)
    u = _shape_field(case, seed)
    # the cells of any seed land in a buffer of one size, their number beside them
    return {"case": case, "ctx": pfc.Context(prob), "u": u, "cells": torch.zeros((u.numel(), 3), device="cuda")}


def _trace32(tr):
    # the trace's sums are of FP32 terms: compared as such
    return tr.astype(np.float32)


def run(s):
    case = s["case"]
    k = case["kind"]
    if k == "grad":
        E, g = s["ctx"].energy_and_grad(s["u"], s["out"])
        return E, g
    if k == "autograd":
        u = s["u"]
        u.grad = None
        E = pfc.PhaseFieldEnergy.apply(u, s["ctx"])
        E.backward()
        return E.detach().float(), u.grad
    if k == "energy":
        return s["ctx"].energy(s["u"])
    if k == "step":
        s["ctx"].step(s["u"], s["out"], TAU, s["scalars"])
        return s["out"]
    if k in ("run", "run_field"):
        s["out"].copy_(s["u"])                      # a run is in place: from this start each time
        tr = s["ctx"].run(s["out"], case["steps"], TAU)
        return s["out"], tr if case.get("prec") == "fp64" else _trace32(tr)
    if k == "batch_step":
        s["batch"].step(s["u"], s["out"], TAU)
        return list(s["out"])
    if k == "batch_run":
        for o, u in zip(s["out"], s["u"]):
            o.copy_(u)
        tr = s["batch"].run(s["out"], case["steps"], TAU)
        return list(s["out"]), _trace32(tr)
    if k == "flow":
        for o, u in zip(s["work"], s["init"]):
            o.copy_(u)
        s["flow"].t = FLOW_T0
        tr = s["flow"].run(*s["work"], case["steps"])
        return list(s["work"]), _trace32(tr)
    if k == "flow_batch":
        for w, t in zip(s["work"], s["init"]):
            for o, u in zip(w, t):
                o.copy_(u)
        s["flow"].t = FLOW_T0
        As, ms, vs = ([w[j] for w in s["work"]] for j in range(3))
        tr = s["flow"].run(As, ms, vs, case["steps"])
        return As, ms, vs, _trace32(tr)
    d = s["ctx"].diagnostics(s["u"])
    k1, k2 = s["ctx"].curvatures(s["u"])
    cells = s["ctx"].surface_cells(s["u"])
    hist = s["ctx"].curvature_histogram(cells, 100, -2.0, 2.0)
    s["cells"][: cells.shape[0]] = cells
    return d, k1, k2, s["cells"], cells.shape[0], hist


# ------------------------------------------------------------------ work

def _step_flops(a):
    """FP32 operations of one voxel's energy, gradient and update (an FMA is two)."""
    return 185.0 if a[0] == a[2] and a[3] == a[4] else 211.0


def work(case):
    k = case["kind"]
    if k == "batch_step":
        return {"bytes": 8.0 * case["n"] ** 3 * case["count"], "flops": 185.0 * case["n"] ** 3 * case["count"]}
    if k == "batch_run":
        N = float(sum(n ** 3 for n, _, _ in _batch_problems(case)))
        return {"bytes": 8.0 * N * case["steps"], "flops": 211.0 * N * case["steps"]}
    N = float(case["nx"]) * case["ny"] * case["nz"]
    if k == "energy":
        return {"bytes": 4.0 * N, "flops": 105.0 * N}
    if k in ("grad", "autograd", "step"):
        return {"bytes": 8.0 * N, "flops": _step_flops(POLYS[case["poly"]]) * N}
    if k == "run":
        b = 16.0 if case["prec"] == "fp64" else 8.0
        return {"bytes": b * N * case["steps"], "flops": _step_flops(POLYS[case["poly"]]) * N * case["steps"]}
    if k == "run_field":
        return {"bytes": 32.0 * N * case["steps"], "flops": 225.0 * N * case["steps"]}
    if k in ("flow", "flow_batch"):
        # A, m, v read and written; the sweep, two blurs of 3 x (2R + 1) taps, div, Adam
        R = math.ceil(3.0 * case["sigma"])
        N *= case["steps"] * case.get("count", 1)
        return {"bytes": 72.0 * N, "flops": (211.0 + 12.0 * (2 * R + 1) + 60.0) * N}
    # diagnostics 4 B, curvatures 12 B, the cells' two passes over u
    return {"bytes": 24.0 * N, "flops": 150.0 * N}


# ------------------------------------------------------------------ exact values, in 64 bits

def _density(u, h, eps, xi, a, well, mu=0.0, theta=None):
    """eq. Feps's density times h^3 of planes 1 .. n-2 of u (n, ny, nx), periodic in x and y;
    a: six numbers, or six arrays of those planes."""
    def sh(t, d, s):                                   # value at +s along axis d (1 y, 2 x)
        return torch.roll(t, -s, d)
    c, up, dn = u[1:-1], u[2:], u[:-2]
    xp, xm, yp, ym = sh(c, 2, 1), sh(c, 2, -1), sh(c, 1, 1), sh(c, 1, -1)
    G = ((xp - xm) / (2 * h), (yp - ym) / (2 * h), (up - dn) / (2 * h))
    H = {(0, 0): (xp + xm - 2 * c) / h**2, (1, 1): (yp + ym - 2 * c) / h**2, (2, 2): (up + dn - 2 * c) / h**2,
         (0, 1): (sh(xp, 1, 1) - sh(xp, 1, -1) - sh(xm, 1, 1) + sh(xm, 1, -1)) / (4 * h**2),
         (0, 2): (sh(up, 2, 1) - sh(up, 2, -1) - sh(dn, 2, 1) + sh(dn, 2, -1)) / (4 * h**2),
         (1, 2): (sh(up, 1, 1) - sh(up, 1, -1) - sh(dn, 1, 1) + sh(dn, 1, -1)) / (4 * h**2)}
    g2 = G[0] ** 2 + G[1] ** 2 + G[2] ** 2
    rho = g2 + xi**2
    q = torch.sqrt(rho)
    w = (c**3 - c if well == 1 else 2 * c * (1 - c) * (1 - 2 * c)) / eps
    M = {k: -eps * v + w * G[k[0]] * G[k[1]] / rho for k, v in H.items()}
    T = M[0, 0] + M[1, 1] + M[2, 2]
    S = M[0, 0] ** 2 + M[1, 1] ** 2 + M[2, 2] ** 2 + 2 * (M[0, 1] ** 2 + M[0, 2] ** 2 + M[1, 2] ** 2)
    a20, a11, a02, a10, a01, a00 = a
    e = (a20 + a02 - a11) / (2 * eps) * S + a11 / (2 * eps) * T**2 + (a10 + a01) / 2 * q * T + a00 * eps * g2
    if not all(isinstance(v, float) for v in a) or a20 != a02 or a10 != a01:
        D = 2 * S - T**2
        P = torch.clamp(D, min=0.0) + xi * torch.log1p(torch.exp(-D.abs() / xi))
        r = torch.where(P > 0, torch.sqrt(torch.where(P > 0, P, torch.ones_like(P))), torch.zeros_like(P))
        e = e + (a20 - a02) / (2 * eps) * T * r + (a10 - a01) / 2 * q * r
    if mu:
        e = e + eps * mu * (theta[0] * G[0] + theta[1] * G[1] + theta[2] * G[2]) ** 2
    return e * h**3


def _evaluate(u, h, eps, xi, a, well, grad=True, mu=0.0, theta=None):
    """(E, dE/du) of a 64-bit field, slab by slab (a: six numbers, or an array (6, nz, ny, nx))."""
    nz = u.shape[0]
    planes = max(1, min(nz, int(6.0e6 / (u.shape[1] * u.shape[2])) or 1))
    E = torch.zeros((), dtype=torch.float64, device=u.device)
    g = torch.empty_like(u) if grad else None
    for z0 in range(0, nz, planes):
        z1 = min(nz, z0 + planes)
        idx = torch.arange(z0 - 2, z1 + 2, device=u.device) % nz       # the densities of z0-1 .. z1 see these
        s = u[idx].detach().requires_grad_(grad)
        ac = tuple(float(v) for v in a) if isinstance(a, tuple) else tuple(f[idx[1:-1]] for f in a)
        e = _density(s, h, eps, xi, ac, well, mu, theta)
        E += e[1:-1].sum().detach()
        if grad:
            (gs,) = torch.autograd.grad(e.sum(), s)
            g[z0:z1] = gs[2:-2]
    return E, g


def _descend(u, steps, tau, trace, ev):
    rows = []
    for _ in range(steps):
        E, g = ev(u)
        lam = g.mean()
        rows.append(torch.stack([E, u.mean(), lam, g.abs().max(), g.abs().mean()]))
        u = u - tau * (g - lam)
    return (u, torch.stack(rows).cpu().numpy()) if trace else u


def _blur(u, sigma):
    R = math.ceil(3.0 * sigma)
    w = [math.exp(-j * j / (2.0 * sigma * sigma)) for j in range(-R, R + 1)]
    t = sum(w)
    for d in (0, 1, 2):
        u = sum(wj / t * torch.roll(u, j, d) for wj, j in zip(w, range(-R, R + 1)))
    return u


def _generate(A, m, v, m0, case):
    h, lr, b1, b2, ae = 0.01, 1e-3, 0.9, 0.999, 1e-8
    A, m, v = A.double(), m.double(), v.double()
    rows = []
    axis = (2, 1, 0)                                   # component c differentiates along x, y, z
    for k in range(case["steps"]):
        t = FLOW_T0 + k + 1
        div = sum(torch.roll(A[c], -1, axis[c]) - torch.roll(A[c], 1, axis[c]) for c in range(3)) / (2 * h) + m0
        E, g = _evaluate(_blur(div, case["sigma"]), h, 0.02, FLOW_XI, PAPER, 1)
        kg = _blur(g, case["sigma"])
        gA = torch.stack([(torch.roll(kg, 1, axis[c]) - torch.roll(kg, -1, axis[c])) / (2 * h) for c in range(3)])
        m = b1 * m + (1 - b1) * gA
        v = b2 * v + (1 - b2) * gA**2
        A = A - lr * (m / (1 - b1**t)) / (torch.sqrt(v / (1 - b2**t)) + ae)
        rows.append(torch.stack([E, gA.abs().max(), gA.abs().mean(), div.mean(), torch.full_like(E, float(t))]))
    return A, m, v, torch.stack(rows).cpu().numpy()


def _analyse(u, eps):
    h = 1.0
    G2 = sum(((torch.roll(u, -1, d) - torch.roll(u, 1, d)) / (2 * h)) ** 2 for d in (0, 1, 2))
    W = 0.25 * (1 - u * u) ** 2 / eps
    dis, ch = float((0.5 * eps * G2 - W).abs().sum()), float((0.5 * eps * G2 + W).sum())
    d = {"discrepancy": dis, "cahn_hilliard": ch, "ratio": dis / ch, "max": float(u.max()), "min": float(u.min())}
    def at(z, y, x):
        return torch.roll(u, (-z, -y, -x), (0, 1, 2))
    e = ((0, 0, 1), (0, 1, 0), (1, 0, 0))              # unit steps along x, y, z as (z, y, x)
    G = [(at(*e[c]) - at(*[-v for v in e[c]])) / 2 for c in range(3)]
    rho = G[0] ** 2 + G[1] ** 2 + G[2] ** 2 + 1e-12
    w = (u**3 - u) / eps
    T, S = 0.0, 0.0
    for i in range(3):
        for j in range(i, 3):
            if i == j:
                H = at(*e[i]) - 2 * u + at(*[-v for v in e[i]])
            else:
                p, q = np.array(e[i]), np.array(e[j])
                H = (at(*map(int, p + q)) - at(*map(int, p - q)) - at(*map(int, q - p)) + at(*map(int, -p - q))) / 4
            M = -eps * H + w * G[i] * G[j] / rho
            T = T + M if i == j else T
            S = S + (1 if i == j else 2) * M * M
    root = torch.sqrt(torch.clamp(2 * S - T * T, min=0.0))
    den = 2 * eps * torch.sqrt(rho)
    return d, (T + root) / den, (T - root) / den


def exact(case, seed):
    k = case["kind"]
    tau = TAU
    if k in ("grad", "autograd", "energy", "step", "run"):
        a = POLYS[case["poly"]]
        ev = lambda u: _evaluate(u, 1.0, case["eps"], case["xi"], a, case.get("well", 0), k != "energy")  # noqa: E731
        u = _field(case, seed).double()
        if k in ("grad", "autograd"):
            E, g = ev(u)
            return E, g
        if k == "energy":
            return ev(u)[0]
        if k == "step":
            return _descend(u, 1, tau, False, ev)
        return _descend(u, case["steps"], tau, True, ev)
    if k == "batch_step":
        return [_descend(u.double(), 1, tau, False,
                         lambda x, a=POLYS[p]: _evaluate(x, 1.0, case["eps"], case["xi"], a, 0))
                for u, (_, p, _) in zip(_batch_fields(case, seed), _batch_problems(case))]
    if k == "batch_run":
        got = [_descend(u.double(), case["steps"], tau, True,
                        lambda x, a=a: _evaluate(x, 1.0, case["eps"], case["xi"], a, 0))
               for u, (_, a, _) in zip(_batch_fields(case, seed), _batch_problems(case))]
        return [u for u, _ in got], np.stack([t for _, t in got])
    if k == "flow":
        A, m, v, tr = _generate(*_flow_state(case, seed, 1)[0], FLOW_M0, case)
        return [A, m, v], tr
    if k == "flow_batch":
        got = [_generate(*s, m0, case) for s, m0 in zip(_flow_state(case, seed, case["count"]),
                                                        _flow_masses(case["count"]))]
        return [g[0] for g in got], [g[1] for g in got], [g[2] for g in got], np.stack([g[3] for g in got])
    if k == "run_field":
        a = _coef_field(case).double()
        u = _noise(_shape(case), 0.3, 0.1, _gen(seed)).double()
        return _descend(u, case["steps"], tau, True,
                        lambda x: _evaluate(x, 1.0, case["eps"], case["xi"], a, 0, mu=MU, theta=THETA))
    # the cells and their histogram are a triangulation, not a formula
    d, k1, k2 = _analyse(_shape_field(case, seed).double(), case["eps"])
    return d, k1, k2, None, None, None
