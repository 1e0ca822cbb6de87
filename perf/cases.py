"""The evaluations this library is timed on, as its users call them.

A case is one call of a public entry point (``FMM.eval``, ``FMM.eval_f32`` or the
differentiable ``fmm_potential``) on seeded synthetic particles.  Callers that
want full accuracy work in float64 with an FP64 plan; callers that accept
single precision hold float32 tensors and a mixed-precision plan.  The
workload shapes are the ones of ``paper_2305_17867_gb300/workloads.py``, with
smaller and ragged relatives of them.
"""
from __future__ import annotations

import math

import torch

from paper_2305_17867_gb300.fmm import FMM, fmm_potential

DEVICE = "cuda"


def _case(name, call, kernel, d, p, levels, n_src, n_tgt, precision, m2l="dense", lam=0.0,
          dist="uniform", grad=False, max_leaf=64):
    """call: "eval" (float64 tensors), "eval_f32" (float32 tensors) or "train"
    (float32, forward and backward); levels < 0: adaptive tree; n_tgt = 0: the
    targets are the sources."""
    return {"name": name, "call": call, "kernel": kernel, "d": d, "p": p, "levels": levels,
            "n_src": n_src, "n_tgt": n_tgt, "precision": precision, "m2l": m2l, "lam": lam,
            "dist": dist, "grad": grad, "max_leaf": max_leaf}


def listed():
    return [
        # the smallest call: a few thousand charges in the plane, full accuracy
        # (one step of a 2D particle or boundary-integral code)
        _case("laplace2d_n2k", "eval", "laplace", 2, 8, 4, 2000, 0, "fp64"),
        # a small 3D system evaluated every time step: latency matters
        _case("laplace3d_n6k", "eval_f32", "laplace", 3, 6, 3, 6007, 0, "f16x3"),
        # potential and forces of an N-body step of ordinary size
        _case("laplace3d_forces_n50k", "eval_f32", "laplace", 3, 8, 4, 50021, 0, "f16x3",
              grad=True),
        # an ordinary large Coulomb evaluation
        _case("laplace3d_n1m", "eval_f32", "laplace", 3, 10, 5, 1_000_000, 0, "f16x3"),
        # a training step through the autograd entry: the potential and the
        # gradients of positions, weights and targets
        _case("laplace3d_train_n1m", "train", "laplace", 3, 8, 5, 1_000_000, 1_000_000, "f16x3"),
        # the largest uniform evaluation (thin-plate / biharmonic kernel)
        _case("biharmonic3d_n4m", "eval_f32", "biharmonic", 3, 8, 6, 4_000_000, 0, "f16x3"),
        # clustered particles on an adaptive tree, separate targets: the largest call
        _case("yukawa3d_adaptive_n2m", "eval_f32", "yukawa", 3, 12, -10, 2_000_000, 2_000_000,
              "bf16x3", lam=1.0, dist="plummer"),
        # the same at the size of a small simulation
        _case("yukawa3d_adaptive_n60k", "eval_f32", "yukawa", 3, 8, -10, 60_013, 60_029,
              "tf32x3", lam=1.0, dist="plummer"),
        # full accuracy in 3D: reference potentials and forces
        _case("laplace3d_fp64_n100k", "eval", "laplace", 3, 10, 4, 100_003, 0, "fp64", "auto",
              grad=True),
        # time-harmonic scattering: complex potential and gradient
        _case("helmholtz3d_n70k", "eval_f32", "helmholtz", 3, 10, 4, 70_001, 0, "tf32x3",
              lam=6.0, grad=True),
        # 2D biharmonic (Stokes-like) potential and gradient at separate targets, full accuracy
        _case("biharmonic2d_fp64_n120k", "eval", "biharmonic", 2, 10, 6, 120_011, 60_007, "fp64",
              "auto", grad=True),
        # screened Coulomb on a uniform tree, plain float arithmetic
        _case("yukawa3d_fp32_n200k", "eval_f32", "yukawa", 3, 12, 4, 200_003, 0, "fp32", "auto",
              lam=1.0),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _levels(rng, n, d, most):
    """A leaf depth that leaves about 8 to 40 points in a leaf."""
    per = math.exp(rng.uniform(math.log(8.0), math.log(40.0)))
    return max(2, min(most, int(round(math.log(max(n / per, 1.0), 2 ** d)))))


def draw(rng):
    kind = rng.choice(["mixed", "mixed", "mixed", "train", "adaptive", "adaptive", "fp64",
                       "fp64_2d", "helmholtz", "fp32"])
    name = ""
    if kind in ("mixed", "train"):
        kernel = rng.choice(["laplace", "biharmonic", "yukawa"])
        n = _log_uniform(rng, 2_000, 4_000_000 if kind == "mixed" else 1_000_000)
        levels = _levels(rng, n, 3, 6 if kind == "mixed" else 5)
        top = {6: 8, 5: 10}.get(levels, 12)
        if kernel == "biharmonic" and levels == 5:
            top = 8
        p = rng.randint(4, top)
        precision = rng.choice(["f16x3", "f16x3", "tf32x3", "bf16x3"])
        if levels == 6 and precision == "tf32x3":
            precision = "f16x3"
        same = kind == "mixed" and rng.random() < 0.6
        return _case(name, "eval_f32" if kind == "mixed" else "train", kernel, 3, p, levels, n,
                     0 if same else max(1, int(n * rng.uniform(0.3, 1.0))), precision, lam=1.0,
                     grad=kind == "mixed" and levels <= 5 and rng.random() < 0.4)
    if kind == "adaptive":
        kernel = rng.choice(["laplace", "yukawa", "biharmonic"])
        precision = rng.choice(["bf16x3", "bf16x3", "tf32x3", "fp32", "fp64"])
        n = _log_uniform(rng, 3_000, {"bf16x3": 1_000_000, "tf32x3": 500_000, "fp32": 60_000,
                                      "fp64": 15_000}[precision])
        p = rng.randint(4, 8 if kernel == "biharmonic" or precision in ("fp32", "fp64") else 12)
        nt = 0 if rng.random() < 0.4 else max(1, int(n * rng.uniform(0.5, 1.0)))
        return _case(name, "eval" if precision == "fp64" else "eval_f32", kernel, 3, p, -10, n, nt,
                     precision, lam=1.0, dist=rng.choice(["plummer", "plummer", "uniform"]),
                     max_leaf=rng.choice([32, 64, 100]))
    if kind == "fp64":
        n = _log_uniform(rng, 1_000, 120_000)
        levels = _levels(rng, n, 3, 4)
        return _case(name, "eval", rng.choice(["laplace", "biharmonic", "yukawa"]), 3,
                     rng.randint(4, 8 if levels == 4 else 10), levels, n,
                     0 if rng.random() < 0.5 else n // 2 + 1, "fp64", "auto", lam=1.0,
                     grad=rng.random() < 0.5)
    if kind == "fp64_2d":
        n = _log_uniform(rng, 500, 200_000)
        return _case(name, "eval", rng.choice(["laplace", "biharmonic"]), 2, rng.randint(6, 14),
                     _levels(rng, n, 2, 6), n, 0 if rng.random() < 0.5 else n // 3 + 1, "fp64",
                     rng.choice(["dense", "auto"]), grad=rng.random() < 0.5)
    if kind == "helmholtz":
        n = _log_uniform(rng, 2_000, 120_000)
        return _case(name, "eval_f32", "helmholtz", 3, rng.randint(6, 10),
                     _levels(rng, n, 3, 4), n, 0 if rng.random() < 0.5 else n // 2 + 1,
                     rng.choice(["tf32x3", "bf16x3"]), lam=rng.uniform(1.0, 6.0),
                     grad=rng.random() < 0.5)
    n = _log_uniform(rng, 2_000, 300_000)
    return _case(name, "eval_f32", rng.choice(["laplace", "yukawa"]), 3, rng.randint(4, 12),
                 _levels(rng, n, 3, 4), n, 0, "fp32", "auto", lam=1.0, grad=rng.random() < 0.3)


# ---- inputs -------------------------------------------------------------------
def _points(gen, n, d, dist, dtype):
    """n points in [0, 1)^d: uniform, or a Plummer sphere of scale 0.1 about the centre."""
    if dist == "uniform":
        return torch.rand(n, d, generator=gen, device=DEVICE, dtype=dtype)
    got, have = [], 0
    while have < n:
        m = int((n - have) * 1.2) + 16
        u = torch.rand(m, generator=gen, device=DEVICE, dtype=torch.float64).clamp(1e-12, 1 - 1e-12)
        v = torch.randn(m, d, generator=gen, device=DEVICE, dtype=torch.float64)
        r = 0.1 / torch.sqrt(u ** (-2.0 / 3.0) - 1.0)
        x = (0.5 + r[:, None] * v / v.norm(dim=1, keepdim=True)).to(dtype)
        x = x[((x >= 0) & (x < 1)).all(dim=1)]
        got.append(x)
        have += x.shape[0]
    return torch.cat(got)[:n].contiguous()


def _inputs(case, seed):
    dtype = torch.float64 if case["call"] == "eval" else torch.float32
    gen = torch.Generator(device=DEVICE).manual_seed(seed)
    ns, nt, d = case["n_src"], case["n_tgt"], case["d"]
    src = _points(gen, ns, d, case["dist"], dtype)
    if case["dist"] == "plummer":
        w = torch.randn(ns, generator=gen, device=DEVICE, dtype=dtype)
    else:
        w = torch.rand(ns, generator=gen, device=DEVICE, dtype=dtype) * 2 - 1
    tgt = _points(gen, nt, d, "uniform", dtype) if nt else None
    u = (torch.randn(nt, generator=gen, device=DEVICE, dtype=dtype)
         if case["call"] == "train" else None)
    return src, w, tgt, u


def prepare(case, seed):
    src, w, tgt, u = _inputs(case, seed)
    plan = FMM(case["kernel"], d=case["d"], p=case["p"], levels=case["levels"], lam=case["lam"],
               precision=case["precision"], m2l=case["m2l"], max_leaf=case["max_leaf"],
               device=DEVICE)
    if case["call"] == "train":
        for t in (src, w, tgt):
            t.requires_grad_(True)
    return {"call": case["call"], "grad": case["grad"], "plan": plan, "src": src, "w": w,
            "tgt": tgt, "u": u}


def run(state):
    plan, src, w, tgt = state["plan"], state["src"], state["w"], state["tgt"]
    if state["call"] == "train":
        phi = fmm_potential(plan, src, w, tgt)
        gs, gw, gt = torch.autograd.grad(phi, (src, w, tgt), state["u"])
        return {"phi": phi.detach(), "grad_src": gs, "grad_w": gw, "grad_tgt": gt}
    entry = plan.eval if state["call"] == "eval" else plan.eval_f32
    out = entry(src, w, tgt, grad=state["grad"])
    return {"phi": out[0], "grad": out[1]} if state["grad"] else {"phi": out}


# ---- what a pass cannot do without ------------------------------------------------
def _stored(d, p, c):
    """Coefficients of a compressed expansion: N(p) - N(p - c)."""
    return math.comb(p + d, d) - (math.comb(p - c + d, d) if p >= c else 0)


def work(case):
    """Inputs read once, outputs written once; the near field's pairs (about 10
    operations each, 8 more for a gradient), the expansions' evaluation at the
    points and the dense translations (2 |j|^2 operations; 8 per frequency in
    their convolution form).  The counts of an adaptive tree are estimates: 8
    translations and 20 near pairs per point, at 64 points a leaf."""
    d, p, ns = case["d"], case["p"], case["n_src"]
    nt = case["n_tgt"] or ns
    c = 4 if case["kernel"] == "biharmonic" else 2
    item = 8 if case["call"] == "eval" else 4
    parts = 2 if case["kernel"] == "helmholtz" else 1
    out = parts * (1 + (d if case["grad"] else 0))
    nbytes = item * (ns * (d + 1) + (case["n_tgt"] * d) + nt * out)
    j, full = _stored(d, p, c), math.comb(p + d, d)
    if case["levels"] < 0:
        m2l = 8.0 * (ns + nt) * 64 / case["max_leaf"]
        pairs = 20.0 * nt * case["max_leaf"] / 64
    else:
        m2l, pairs = 0.0, 0.0
        for lev in range(2, case["levels"] + 1):
            n = 1 << lev
            near = 3 * n - 2
            listed_ = sum(min(2 * (t // 2) + 3, n - 1) - max(2 * (t // 2) - 2, 0) + 1
                          for t in range(n))
            m2l += listed_ ** d - near ** d
        pairs = ns * nt * (near / float(n * n)) ** d
    if case["m2l"] == "auto" and case["levels"] > 0:
        per = 8.0 * (p + 1) * (2 * p + 1) ** (d - 2) * (2 * min(c, p + 1) - 1)
    else:
        per = 2.0 * j * j
    flops = parts * m2l * per + pairs * parts * (10 + (8 if case["grad"] else 0))
    flops += 2.0 * full * (ns + parts * nt * (1 + (d if case["grad"] else 0)))
    if case["call"] == "train":  # grad phi with phi, then the transposed evaluation
        nbytes += item * (nt + ns * (1 + d) + nt * d)
        flops = 2 * flops + 8 * 2 * pairs + 2.0 * full * d * (ns + nt)
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---- the same sums, pair by pair in 64 bits ----------------------------------------
def _radial(kernel, d, lam, r, grad):
    """G(r) and, for the gradient, G'(r) / r."""
    if kernel == "laplace" and d == 2:
        return torch.log(r), 1 / (r * r) if grad else None
    if kernel == "laplace":
        g = 1 / (4 * math.pi * r)
        return g, -g / (r * r) if grad else None
    if kernel == "biharmonic" and d == 2:
        lg = torch.log(r)
        return r * r * lg, 2 * lg + 1 if grad else None
    if kernel == "biharmonic":
        return r, 1 / r if grad else None
    k = 1j * lam if kernel == "helmholtz" else -lam
    g = torch.exp(k * r) / r
    return g, g * (k * r - 1) / (r * r) if grad else None


def _direct(case, src, w, tgt, grad):
    """phi (and grad phi) at tgt; pairs at distance zero are skipped."""
    kernel, lam, ns, nt = case["kernel"], case["lam"], src.shape[0], tgt.shape[0]
    cplx = kernel == "helmholtz"
    wc = w.to(torch.complex128) if cplx else w
    phi = torch.zeros(nt, dtype=wc.dtype, device=DEVICE)
    g = torch.zeros(nt, case["d"], dtype=wc.dtype, device=DEVICE) if grad else None
    step = max(1, (1 << 25) // max(ns, 1))
    for a in range(0, nt, step):
        x = tgt[a:a + step]
        dx = [x[:, k, None] - src[None, :, k] for k in range(case["d"])]
        r = torch.sqrt(sum(v * v for v in dx))
        same = r == 0
        r.masked_fill_(same, 1.0)
        val, dr = _radial(kernel, case["d"], lam, r, grad)
        phi[a:a + step] = val.masked_fill(same, 0.0) @ wc
        if grad:
            dr = dr.masked_fill(same, 0.0) * wc
            for k in range(case["d"]):
                g[a:a + step, k] = (dr * dx[k]).sum(dim=1)
    return phi, g


def exact(case, seed):
    nt = case["n_tgt"] or case["n_src"]
    cost = float(case["n_src"]) * nt
    cost *= 3.0 if case["grad"] else 1.0
    cost *= 6.0 if case["call"] == "train" else 1.0
    cost *= {"helmholtz": 4.0, "yukawa": 1.5}.get(case["kernel"], 1.0)
    if cost > 7e10:
        return None
    src, w, tgt, u = (None if t is None else t.double() for t in _inputs(case, seed))
    tgt = src if tgt is None else tgt
    if case["call"] != "train":
        phi, g = _direct(case, src, w, tgt, case["grad"])
        return {"phi": phi, "grad": g} if case["grad"] else {"phi": phi}
    phi, gphi = _direct(case, src, w, tgt, True)
    psi, gpsi = _direct(case, tgt, u, src, True)
    return {"phi": phi, "grad_src": w[:, None] * gpsi, "grad_w": psi,
            "grad_tgt": u[:, None] * gphi}
