"""Timed cases: the work that programs have this library do, through its public entry points.

A case is a dict of plain values; ``listed()`` gives the fixed ones, ``draw()``
more of the same ranges.  ``prepare`` makes what a program holds before the
call (solver, batch, tables), ``run`` is one call of such a program, ``work``
the bytes and operations it cannot do without, and ``exact`` the same result
in FP64, computed here from the method's definition with torch (dense
advected-basis matrices, inverted; the reduced form of the constrained least
squares) without the library's code.

Results come back in the precision of the mode: FP64 runs return the FP64
moments as they are, FP32 and mixed runs hand them on in single precision.
"""

from __future__ import annotations

import math

import numpy as np
import torch

import paper_2009_07340_gb300 as sl

PI = math.pi
DEV = "cuda"


# ---------------------------------------------------------------- the cases
def listed():
    return [
        # the smallest call: one whole small solve (1D constant drift-diffusion,
        # a Gaussian pulse, 256 samples, 100 steps), created, advanced, averaged
        # to the host and freed, as a served request or a parameter study does
        {"name": "solve_1d_small_fp64", "kind": "solve", "dim": 1, "precision": "fp64", "K": 8, "N": 6, "M": 256,
         "steps": 100, "dt": 1.0, "rule": "edge", "flow": "const"},
        # many small uneven 1D solves advanced together, moments of each to the
        # host: ensembles and parameter studies
        {"name": "batch_1d_small_fp32", "kind": "batch", "dim": 1, "precision": "fp32", "count": 32, "Klo": 8,
         "Khi": 64, "Nlo": 4, "Nhi": 8, "Mlo": 16, "Mhi": 128, "steps": 100},
        # the headline: 256 elements of the highest order, 4096 samples, resident
        # state, a slice of its time steps and the sample moments
        {"name": "steps_1d_n16_fp32", "kind": "steps", "dim": 1, "precision": "fp32", "K": 256, "N": 16, "M": 4096,
         "steps": 50, "dt": 0.5, "rule": "node", "flow": "sin"},
        # an odd order on a mesh above 256 elements (one sample spans several
        # thread blocks), an odd sample count, the mixed precision form
        {"name": "steps_1d_n11_mixed", "kind": "steps", "dim": 1, "precision": "mixed", "K": 777, "N": 11, "M": 501,
         "steps": 30, "dt": 0.5, "rule": "node", "flow": "sin"},
        # the default precision on an ordinary mesh: reference runs
        {"name": "steps_1d_n8_fp64", "kind": "steps", "dim": 1, "precision": "fp64", "K": 256, "N": 8, "M": 1024,
         "steps": 10, "dt": 0.5, "rule": "node", "flow": "sin"},
        # few elements, many samples, Dirichlet boundary values per step and
        # reseeding: the shape of the paper's own 1D tests
        {"name": "steps_1d_dirichlet_fp32", "kind": "dirichlet", "dim": 1, "precision": "fp32", "K": 20, "N": 9,
         "M": 10000, "steps": 100, "reseed": 50, "dt": 0.5, "rule": "node", "flow": "const"},
        # statistics of samples in hand: moments and the PDF at every node
        {"name": "statistics_1d_fp32", "kind": "statistics", "dim": 1, "precision": "fp32", "K": 200, "N": 7,
         "M": 4001, "bins": 64},
        # 2D solid-body rotation with variable diffusion on 64 x 64 elements
        {"name": "steps_2d_n8_fp32", "kind": "steps", "dim": 2, "precision": "fp32", "K": 64, "Ky": 64, "N": 8,
         "M": 64, "steps": 2, "dt": 0.5, "rule": "node", "flow": "rotation"},
        # uneven 2D solves in the mixed form, one step, moments to the host
        {"name": "batch_2d_mixed", "kind": "batch", "dim": 2, "precision": "mixed", "count": 12, "Klo": 16, "Khi": 64,
         "Nlo": 4, "Nhi": 12, "Mlo": 4, "Mhi": 32, "steps": 1},
        # 2D in the default precision
        {"name": "steps_2d_n6_fp64", "kind": "steps", "dim": 2, "precision": "fp64", "K": 32, "Ky": 32, "N": 6,
         "M": 32, "steps": 1, "dt": 0.5, "rule": "edge", "flow": "rotation"},
        # the highest 2D order on an uneven mesh with odd sizes
        {"name": "steps_2d_n12_fp32", "kind": "steps", "dim": 2, "precision": "fp32", "K": 19, "Ky": 23, "N": 12,
         "M": 101, "steps": 1, "dt": 0.5, "rule": "edge", "flow": "const"},
        # coupled to a field solver on the same GPU: a new nodal drift and
        # diffusion (device tables) before every step
        {"name": "coupled_2d_n5_fp32", "kind": "coupled", "dim": 2, "precision": "fp32", "K": 32, "Ky": 32, "N": 5,
         "M": 64, "steps": 2, "dt": 0.5, "rule": "edge"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# seconds that a pass of this many element-sample updates may be expected to
# take at most (only to keep drawn cases below the largest listed one)
def _seconds(dim, N, precision, esu):
    ops = 6 * N * N + 22 * N if dim == 1 else 500 * N * N * (1 + N / 6)
    rate = {"fp32": 2e13, "mixed": 1e13, "fp64": 3e11}[precision]
    return esu * ops / (rate if dim == 1 else 0.25 * rate)


def _cap(c, E, esu_per_sample):
    """The case with its sample count reduced until a pass costs at most ~6 ms."""
    per = _seconds(c["dim"], c["N"], c["precision"], esu_per_sample)
    c["M"] = max(3, min(c["M"], int(6e-3 / per), 1 + (1 << 24) // (E * c["N"] ** c["dim"])))
    return c


def draw(rng):
    kind = rng.choice(["solve", "steps1", "steps1", "steps1", "steps2", "steps2", "steps2", "dirichlet", "statistics",
                       "batch1", "batch2", "coupled"])
    prec = rng.choice(["fp32", "fp32", "mixed", "fp64"])
    if kind == "solve":
        c = {"kind": "solve", "dim": 1, "precision": rng.choice(["fp64", "fp32"]), "K": _log(rng, 4, 40),
             "N": rng.randint(4, 9), "M": _log(rng, 64, 1000), "steps": rng.randint(20, 120), "dt": 1.0,
             "rule": "edge", "flow": "const"}
        return _cap(c, c["K"], c["K"] * c["steps"])
    if kind == "steps1":
        c = {"kind": "steps", "dim": 1, "precision": prec, "K": _log(rng, 8, 1024), "N": rng.randint(4, 16),
             "M": _log(rng, 100, 4096), "steps": rng.randint(10, 50), "dt": 0.5, "rule": "node", "flow": "sin"}
        if prec != "mixed" and rng.random() < 0.2 and c["K"] * c["N"] * c["M"] < 1 << 20:
            c["components"] = 2
        return _cap(c, c["K"], c["K"] * c["steps"])
    if kind == "steps2":
        c = {"kind": "steps", "dim": 2, "precision": prec, "K": rng.randint(16, 64), "Ky": rng.randint(16, 64),
             "N": rng.randint(4, 11 if prec == "fp64" else 12), "M": _log(rng, 8, 64), "steps": 1, "dt": 0.5,
             "rule": "edge", "flow": rng.choice(["const", "rotation"])}
        if c["N"] <= 8 and rng.random() < 0.3:
            c["rule"], c["dt"] = "node", 0.4
        if c["N"] <= 8 and rng.random() < 0.2:
            c["components"], c["M"] = 2, min(c["M"], 16)
        return _cap(c, c["K"] * c["Ky"], c["K"] * c["Ky"] * (1 + 0.5 * (c.get("components", 1) - 1)))
    if kind == "dirichlet":
        c = {"kind": "dirichlet", "dim": 1, "precision": rng.choice(["fp32", "fp64"]), "K": _log(rng, 3, 64),
             "N": rng.randint(4, 16), "M": _log(rng, 500, 10000), "steps": rng.randint(20, 100),
             "reseed": rng.choice([0, 10, 25]), "dt": 0.5, "rule": "node", "flow": "const"}
        return _cap(c, c["K"], c["K"] * c["steps"])
    if kind == "statistics":
        c = {"kind": "statistics", "dim": 1, "precision": rng.choice(["fp32", "fp64"]), "K": _log(rng, 16, 256),
             "N": rng.randint(4, 16), "M": _log(rng, 500, 4001), "bins": rng.choice([16, 50, 64, 100])}
        c["M"] = min(c["M"], 6_000_000 // (c["K"] * c["N"]))
        return c
    if kind == "batch1":
        return {"kind": "batch", "dim": 1, "precision": rng.choice(["fp32", "mixed"]), "count": rng.randint(8, 32),
                "Klo": 8, "Khi": rng.randint(40, 64), "Nlo": 4, "Nhi": rng.randint(8, 12), "Mlo": 16,
                "Mhi": rng.randint(64, 128), "steps": rng.randint(20, 100)}
    if kind == "batch2":
        return {"kind": "batch", "dim": 2, "precision": rng.choice(["fp32", "mixed"]), "count": rng.randint(4, 10),
                "Klo": 16, "Khi": rng.randint(30, 56), "Nlo": 4, "Nhi": rng.randint(8, 12), "Mlo": 4,
                "Mhi": rng.randint(8, 24), "steps": 1}
    c = {"kind": "coupled", "dim": 2, "precision": rng.choice(["fp32", "fp64"]), "K": rng.randint(12, 48),
         "Ky": rng.randint(12, 48), "N": rng.randint(4, 9), "M": _log(rng, 8, 64), "steps": rng.randint(1, 2),
         "dt": 0.5, "rule": "edge"}
    return _cap(c, c["K"] * c["Ky"], c["K"] * c["Ky"] * c["steps"])


# ------------------------------------------------------------ the problems
def _nodes(N):
    return 0.5 * (1.0 - np.cos((np.arange(N) + 0.5) * PI / N))


def _u_at(spec, x, y):
    kind, p = spec
    if kind == "const":
        return [p[0] + 0 * x, p[1] + 0 * x]
    if kind == "sin":
        return [p[0] + p[1] * np.sin(p[2] * PI * x), 0 * x]
    return [-p[0] * (y - p[2]), p[0] * (x - p[1])]


def _d_at(spec, x, y):
    kind, p = spec
    if kind == "const":
        return p[0] + 0 * x
    if kind == "cos":
        return p[0] * (1 + p[1] * np.cos(p[2] * PI * x))
    return p[0] * (1 + p[1] * np.sin(p[2] * PI * x) * np.sin(p[3] * PI * y))


def _phi_at(spec, pb, x, y):
    kind, p = spec
    if kind == "fourier":
        v = p[0] + 0 * x
        for k in range(1, int(p[2]) + 1):
            v = v + p[1 + 2 * k] * np.cos(k * p[1] * PI * x) + p[2 + 2 * k] * np.sin(k * p[1] * PI * x)
        return v
    v = 0 * x
    for ix in (-1, 0, 1):
        for iy in (-1, 0, 1) if pb["dim"] == 2 else (0,):
            r2 = (x - p[2] + ix * (pb["hi"][0] - pb["lo"][0])) ** 2
            if pb["dim"] == 2:
                r2 = r2 + (y - p[3] + iy * (pb["hi"][1] - pb["lo"][1])) ** 2
            v = v + np.exp(-r2 / (2 * p[1] ** 2))
    return p[0] * v


def _coords(pb):
    """Node coordinates (x, y), flat in the state's order [E][N^dim]."""
    xi, N = _nodes(pb["N"]), pb["N"]
    h = [(pb["hi"][d] - pb["lo"][d]) / pb["K"][d] for d in range(pb["dim"])]
    gx = pb["lo"][0] + (np.arange(pb["K"][0])[:, None] + xi) * h[0]
    if pb["dim"] == 1:
        return gx.ravel(), 0 * gx.ravel()
    gy = pb["lo"][1] + (np.arange(pb["K"][1])[:, None] + xi) * h[1]
    shape = (pb["K"][1], pb["K"][0], N, N)  # ky, kx, j, i
    x = np.broadcast_to(gx[None, :, None, :], shape)
    y = np.broadcast_to(gy[:, None, :, None], shape)
    return x.ravel().copy(), y.ravel().copy()


def _bound(pb, u, D, rule):
    """Largest dt with |u| dt + sqrt(2 D dt) <= gap in every direction: the
    smallest node gap ("node") or the first node's distance to the face ("edge")."""
    xi = _nodes(pb["N"])
    gap = float(np.diff(xi).min()) if rule == "node" else float(xi[0])
    b, best = math.sqrt(2 * float(np.max(D))), math.inf
    for d in range(pb["dim"]):
        dx, um = gap * (pb["hi"][d] - pb["lo"][d]) / pb["K"][d], float(np.max(np.abs(u[d])))
        s = dx / b if um == 0 else (-b + math.sqrt(b * b + 4 * um * dx)) / (2 * um)
        best = min(best, s * s)
    return best


def _fourier(rng, modes=8):
    ab = rng.uniform(-1, 1, size=(modes, 2))
    ab *= 0.5 / np.abs(ab).sum()
    return ("fourier", [1.0, 1.0, float(modes)] + [float(v) for v in ab.ravel()])


def _problem(c, seed):
    """The problem of a single-solver case: its fields and time step from the seed."""
    rng = np.random.default_rng([17, seed])
    dim = c["dim"]
    L = 2.0 if dim == 1 else 1.0
    pb = {"dim": dim, "K": (c["K"],) if dim == 1 else (c["K"], c["Ky"]), "lo": (0.0,) * dim, "hi": (L,) * dim,
          "N": c["N"], "M": c["M"], "steps": c.get("steps", 1), "seed": int(seed) * 7919 + 3}
    if c.get("flow", "const") == "sin":
        pb["drift"] = ("sin", [1.0 + 0.1 * rng.uniform(-1, 1), 0.5, 1.0])
        pb["diffusion"] = ("cos", [0.01, 0.5, 1.0])
    elif c.get("flow", "const") == "rotation":
        pb["drift"] = ("rotation", [2 * PI * (1 + 0.05 * rng.uniform(-1, 1)), 0.5, 0.5])
        pb["diffusion"] = ("sinsin", [0.005, 0.3, 2.0, 2.0])
    else:
        pb["drift"] = ("const", [float(v) for v in rng.uniform(0.5, 1.0, size=2)])
        pb["diffusion"] = ("const", [0.01 if dim == 1 else float(rng.uniform(1e-3, 1e-2))])
    if dim == 2:
        pb["phi0"] = ("gauss", [1.0, 0.05] + [float(v) for v in rng.uniform(0.35, 0.65, size=2)])
    elif c["kind"] == "solve":
        pb["phi0"] = ("gauss", [1.0, 0.1, float(rng.uniform(0.8, 1.2)), 0.0])
    else:
        pb["phi0"] = _fourier(rng)
    x, y = _coords(pb)
    if c["kind"] == "coupled":
        pb["tables"] = _tables(pb, rng, x, y)
        u, D = [np.stack([t[0][d] for t in pb["tables"]]) for d in (0, 1)], np.stack([t[1] for t in pb["tables"]])
    else:
        u, D = _u_at(pb["drift"], x, y), _d_at(pb["diffusion"], x, y)
    if "dt" in c:
        pb["dt"] = c["dt"] * _bound(pb, u, D, c["rule"])
    if c["kind"] == "dirichlet":
        pb["periodic"] = False
        pb["reseed_every"] = c["reseed"]
        t = np.arange(1, pb["steps"] + 1) * pb["dt"]
        ends = [float(_phi_at(pb["phi0"], pb, np.array([v]), np.zeros(1))[0]) for v in (0.0, L)]
        pb["ghost"] = np.stack([v * (1 + 0.01 * np.sin(40.0 * t + k)) for k, v in enumerate(ends)], axis=1)
    if c.get("components", 1) == 2:
        pb["components"] = 2
        second = ("gauss", [1.0, 0.08] + [float(v) for v in rng.uniform(0.4, 0.6, size=2)]) if dim == 2 else _fourier(rng)
        pb["phi0_2"] = second
    return pb


def _tables(pb, rng, x, y):
    """Nodal drift [2][E n] and diffusion [E n] of two moments of a cellular flow."""
    out = []
    for k in range(2):
        a, b = rng.uniform(0.8, 1.2, size=2)
        ux = a * np.sin(2 * PI * x) * np.cos(2 * PI * y) + 0.3 + 0.1 * k
        uy = -b * np.cos(2 * PI * x) * np.sin(2 * PI * y) - 0.2
        out.append((np.stack([ux, uy]), 0.004 * (1 + 0.3 * np.sin(2 * PI * (x + 0.1 * k)) * np.cos(2 * PI * y))))
    return out


def _instances(c, seed):
    """The uneven instances of a batch: sizes from the case, fields from the seed."""
    rs = np.random.default_rng([5, c["count"], c["Khi"], c["Nhi"], c["Mhi"]])  # sizes: the same for every seed
    out = []
    for i in range(c["count"]):
        K, N = int(rs.integers(c["Klo"], c["Khi"] + 1)), int(rs.integers(c["Nlo"], c["Nhi"] + 1))
        one = {"kind": "batch", "dim": c["dim"], "K": K, "Ky": K, "N": N, "M": int(rs.integers(c["Mlo"], c["Mhi"] + 1)),
               "steps": c["steps"], "dt": 0.5, "rule": "node" if c["dim"] == 1 else "edge",
               "flow": "sin" if c["dim"] == 1 else ("rotation" if rs.random() < 0.5 else "const")}
        pb = _problem(one, int(seed) * 64 + i)
        if c["dim"] == 2:
            pb["diffusion"] = ("const", [float(np.random.default_rng([3, seed, i]).uniform(1e-3, 1e-2))])
            x, y = _coords(pb)
            pb["dt"] = 0.5 * _bound(pb, _u_at(pb["drift"], x, y), _d_at(pb["diffusion"], x, y), "edge")
        out.append(pb)
    return out


def _sample_values(c, seed):
    """Samples in hand for the statistics: a smooth field, scaled and shifted per sample."""
    pb = _problem(c, seed)
    rng = np.random.default_rng([29, seed])
    x, _ = _coords(pb)
    f = _phi_at(pb["phi0"], pb, x, 0 * x)
    g = np.cos(PI * x + rng.uniform(0, 6))
    z = rng.normal(size=(2, pb["M"]))
    return pb, f[None] * (1 + 0.05 * z[0])[:, None] + 0.1 * z[1][:, None] * g[None]


# ------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind, prec = case["kind"], case["precision"]
    if kind == "solve":
        return {"case": case, "pb": _problem(case, seed)}
    if kind == "batch":
        pbs = _instances(case, seed)
        return {"case": case, "batch": sl.Batch(pbs, prec)}
    if kind == "statistics":
        pb, q = _sample_values(case, seed)
        pb["dt"] = 1e-6
        s = sl.Solver(pb, prec)
        s.set_samples(0, q)
    else:
        pb = _problem(case, seed)
        s = sl.Solver(pb, prec)
        if pb.get("components", 1) == 2:  # its second field
            x, y = _coords(pb)
            both = np.stack([_phi_at(pb["phi0"], pb, x, y), _phi_at(pb["phi0_2"], pb, x, y)])
            s.set_samples(0, np.broadcast_to(both.ravel(), (pb["M"], both.size)))
    st = {"case": case, "pb": pb, "solver": s,
          "mean": torch.empty(s.V, dtype=torch.float64, device=DEV),
          "m2": torch.empty(s.V, dtype=torch.float64, device=DEV)}
    if kind == "coupled":
        st["tables"] = [(torch.from_numpy(u.ravel()).to(DEV), torch.from_numpy(D).to(DEV)) for u, D in pb["tables"]]
    return st


def run(state):
    case = state["case"]
    kind, single = case["kind"], case["precision"] != "fp64"
    if kind == "solve":
        with sl.Solver(state["pb"], case["precision"]) as s:
            s.step()
            mean, m2 = s.moments()
        return {"mean": mean.astype(np.float32), "m2": m2.astype(np.float32)} if single else {"mean": mean, "m2": m2}
    if kind == "batch":
        b = state["batch"]
        b.step(case["steps"])
        got = [b.moments(i) for i in range(case["count"])]
        return [tuple(v.astype(np.float32) for v in mm) for mm in got] if single else got
    s, mean, m2 = state["solver"], state["mean"], state["m2"]
    if kind == "statistics":
        s.moments_device(mean, m2)
        lo, hi = 0.0, 2.0
        return {"mean": mean, "m2": m2, "pdf": s.pdf(case["bins"], lo, hi).view(np.int32)}
    if kind == "coupled":
        for k in range(case["steps"]):
            u, D = state["tables"][k % 2]
            s.set_fields_device(("nodal", u), ("nodal", D))
            s.step(steps=1)
    else:
        if kind == "dirichlet":
            s.set_boundary(state["pb"]["ghost"])
        s.step()
    s.moments_device(mean, m2)
    return {"mean": mean.float(), "m2": m2.float()} if single else {"mean": mean, "m2": m2}


# ---------------------------------------------------------------- the work
def _work_one(dim, K, Ky, N, M, steps, precision, comps=1):
    """State in and out once, one increment per sample, step and dimension, the
    moments out; operations: 1D the reduced form (6 N^2 + 8 N, of which a second
    field shares all but 2 N^2 + 8 N); 2D the dense rows applied once to form the
    interpolant and once each way in the least squares (6 n^2), the face rows
    (16 N^2) and the particles' basis (8 N n)."""
    E, n = K * (Ky if dim == 2 else 1), N ** dim
    ops = 6 * N * N + 8 * N + (comps - 1) * (2 * N * N + 8 * N) if dim == 1 else \
        comps * (6 * n * n + 16 * N * N) + 8 * N * n
    return {"bytes": 2 * 8 * M * E * n * comps + 8 * M * steps * dim + 16 * E * n * comps, "flops": ops * E * M * steps}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        one = [_work_one(pb["dim"], pb["K"][0], pb["K"][-1], pb["N"], pb["M"], case["steps"], case["precision"])
               for pb in _instances(case, 0)]
        return {k: sum(w[k] for w in one) for k in ("bytes", "flops")}
    if kind == "statistics":
        V = case["K"] * case["N"]
        return {"bytes": 8 * case["M"] * V + 16 * V + 4 * V * case["bins"], "flops": 6 * case["M"] * V}
    w = _work_one(case["dim"], case["K"], case.get("Ky", 1), case["N"], case["M"], case["steps"], case["precision"],
                  case.get("components", 1))
    if kind == "solve":  # the state is created by the call
        w["bytes"] = 8 * case["M"] * case["steps"] + 16 * case["K"] * case["N"]
    if kind == "coupled":
        w["bytes"] += 24 * case["K"] * case["Ky"] * case["N"] ** 2 * case["steps"]
    return w


# ------------------------------------------------------------------- exact
def _philox(step, sample, seed):
    """The four words of Philox4x32-10 at counter (step, sample, 0, 0)."""
    m32 = np.uint64(0xFFFFFFFF)
    step, sample = np.broadcast_arrays(step, sample)
    c = [step.astype(np.uint64) & m32, sample.astype(np.uint64) & m32, np.zeros(step.shape, np.uint64),
         np.zeros(step.shape, np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, (seed >> 32) & 0xFFFFFFFF
    for _ in range(10):
        p0, p1 = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(p1 >> np.uint64(32)) ^ c[1] ^ np.uint64(k0), p1 & m32, (p0 >> np.uint64(32)) ^ c[3] ^ np.uint64(k1), p0 & m32]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return c


def _wiener(pb, steps, first=0):
    """dW [steps][M][2] (Box-Muller on two 52-bit uniforms)."""
    w = _philox(np.arange(first, first + steps)[:, None], np.arange(pb["M"])[None, :], pb["seed"])
    s32, s12 = np.uint64(32), np.uint64(12)
    u = [(2.0 * (((w[2 * k] << s32) | w[2 * k + 1]) >> s12).astype(np.float64) + 1.0) * 2.0 ** -53 for k in (0, 1)]
    r = np.sqrt(-2.0 * np.log(u[0]))
    return math.sqrt(pb["dt"]) * np.stack([r * np.cos(2 * PI * u[1]), r * np.sin(2 * PI * u[1])], axis=-1)


def _t(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device=DEV)


class _Ref:
    """The method in FP64 for one problem."""

    def __init__(self, pb):
        self.pb, self.dim, self.N = pb, pb["dim"], pb["N"]
        N, dim = self.N, self.dim
        xi = _nodes(N)
        z = xi[:, None] - xi[None, :]
        lam = np.array([1.0 / np.prod([z[j, m] for m in range(N) if m != j]) for j in range(N)])
        self.K = pb["K"] if dim == 2 else (pb["K"][0], 1)
        self.E, self.n = self.K[0] * self.K[1], N ** dim
        self.h = [(pb["hi"][d] - pb["lo"][d]) / pb["K"][d] for d in range(dim)]
        diff = np.zeros((N, N))  # d h_m / d xi at node i
        for i in range(N):
            for m in range(N):
                if i != m:
                    diff[i, m] = lam[m] / lam[i] / z[i, m]
        diff[np.arange(N), np.arange(N)] = -diff.sum(1)
        self.diff, self.z, self.lam = diff, _t(z), _t(lam)
        hb = [np.array([lam[m] * np.prod([x - xi[k] for k in range(N) if k != m]) for m in range(N)]) for x in (0.0, 1.0)]
        self.hb = hb
        B = np.zeros((2, N)) if dim == 1 else np.zeros((4, N, N, N))  # side, point, j, i
        if dim == 1:
            B[0], B[1] = hb
        else:
            for f in range(N):
                B[0, f, f, :], B[1, f, f, :] = hb
                B[2, f, :, f], B[3, f, :, f] = hb
        self.B = _t(B.reshape(-1, self.n))
        if pb.get("tables") is None:
            self.set_fields(None, None)

    def set_fields(self, u, D):
        """Node and face coefficients: analytic fields, or nodal u [2][E n] and D [E n]."""
        pb, N, dim, K = self.pb, self.N, self.dim, self.K
        x, y = _coords(pb)
        nodal = u is not None
        if not nodal:
            u, D = _u_at(pb["drift"], x, y), _d_at(pb["diffusion"], x, y)
        if dim == 1:
            g = np.asarray(u[0]).reshape(K[0], N)
            div = g @ self.diff.T / self.h[0]
            xf = pb["lo"][0] + np.arange(K[0] + 1) * self.h[0]
            uf, Df = _u_at(pb["drift"], xf, 0 * xf)[0], _d_at(pb["diffusion"], xf, 0 * xf)
            if pb.get("periodic", True):
                uf[-1], Df[-1] = uf[0], Df[0]
            self.uf, self.bf = [_t(uf)], [_t(np.sqrt(2 * Df))]
        else:
            g = [np.asarray(v).reshape(K[1], K[0], N, N) for v in u]  # ky kx j i
            Dg = np.asarray(D).reshape(K[1], K[0], N, N)
            div = np.einsum("im,yxjm->yxji", self.diff, g[0]) / self.h[0] + \
                np.einsum("jm,yxmi->yxji", self.diff, g[1]) / self.h[1]
            xi = _nodes(N)
            if nodal:
                def iface(v, ax):
                    e = "f,yxjf->yxj" if ax == 0 else "f,yxfi->yxi"
                    return 0.5 * (np.einsum(e, self.hb[0], v) + np.roll(np.einsum(e, self.hb[1], v), 1, axis=1 - ax))
                uf = [iface(g[0], 0), iface(g[1], 1)]
                Df = [np.maximum(iface(Dg, 0), 0), np.maximum(iface(Dg, 1), 0)]
            else:
                ex = pb["lo"][0] + np.arange(K[0]) * self.h[0]
                ey = pb["lo"][1] + np.arange(K[1]) * self.h[1]
                shape = (K[1], K[0], N)
                pts = [(np.broadcast_to(ex[None, :, None], shape), np.broadcast_to(ey[:, None, None] + xi * self.h[1], shape)),
                       (np.broadcast_to(ex[None, :, None] + xi * self.h[0], shape), np.broadcast_to(ey[:, None, None], shape))]
                uf = [_u_at(pb["drift"], *pts[d])[d] for d in (0, 1)]
                Df = [_d_at(pb["diffusion"], *p) for p in pts]
            self.uf, self.bf = [_t(v) for v in uf], [_t(np.sqrt(2 * v)) for v in Df]
        self.u = [_t(np.asarray(v).reshape(self.E, self.n)) for v in u[:dim]]
        self.b = _t(np.sqrt(2 * np.asarray(D)).reshape(self.E, self.n))
        self.div = _t(div.reshape(self.E, self.n))

    def basis(self, z, d):
        """h_i at node + d: [..., n] displacements -> [..., n, N]."""
        f = z + d[..., None]
        one = torch.ones_like(f[..., :1])
        pre = torch.cumprod(torch.cat([one, f[..., :-1]], -1), -1)
        suf = torch.flip(torch.cumprod(torch.cat([one, torch.flip(f[..., 1:], [-1])], -1), -1), [-1])
        return pre * suf * self.lam

    def step(self, Q, dW, ghost=None):
        """One step of the samples Q [S][comps][E][n], increments dW [S][2]."""
        pb, N, K, dt, S = self.pb, self.N, self.K, self.pb["dt"], Q.shape[0]
        dW = _t(dW)
        disp = [(self.u[d] * dt + self.b * dW[:, d, None, None]) / self.h[d] for d in range(self.dim)]
        if self.dim == 1:
            V = self.basis(self.z, disp[0])
        else:
            zx = self.z.repeat(N, 1)
            zy = self.z.repeat_interleave(N, 0)
            V = (self.basis(zy, disp[1])[..., :, None] * self.basis(zx, disp[0])[..., None, :]).reshape(S, self.E, self.n, self.n)
        Vi = torch.linalg.inv(V)
        del V
        Em = self.B @ Vi  # [S][E][faces][n]
        C = Em @ Em.transpose(-1, -2)
        C.diagonal(dim1=-2, dim2=-1).add_(1.0)
        ps = (Q - dt * self.div * Q).transpose(1, 2).transpose(2, 3)  # [S][E][n][comps]
        F = Em @ ps
        sig = [self.uf[d] * dt + self.bf[d] * dW[:, d].reshape([S] + [1] * self.uf[d].dim()) for d in range(self.dim)]
        if self.dim == 1:
            left, right = torch.roll(F[:, :, 1], 1, 1), torch.roll(F[:, :, 0], -1, 1)
            if not pb.get("periodic", True):
                left[:, 0], right[:, -1] = float(ghost[0]), float(ghost[1])
            pos = (sig[0] > 0)[..., None]
            g = torch.stack([torch.where(pos[:, :-1], left, F[:, :, 0]), torch.where(pos[:, 1:], F[:, :, 1], right)], 2)
        else:
            f = F.reshape(S, K[1], K[0], 4, N, -1)
            gx = torch.where((sig[0] > 0)[..., None], torch.roll(f[:, :, :, 1], 1, 2), f[:, :, :, 0])
            gy = torch.where((sig[1] > 0)[..., None], torch.roll(f[:, :, :, 3], 1, 1), f[:, :, :, 2])
            g = torch.stack([gx, torch.roll(gx, -1, 2), gy, torch.roll(gy, -1, 1)], 3).reshape(F.shape)
        mu = torch.linalg.solve(C, F - g)
        return (Vi @ (ps - Em.transpose(-1, -2) @ mu)).transpose(2, 3).transpose(1, 2).contiguous()


def _exact_one(pb, steps):
    """Mean and second moment after `steps` steps."""
    ref = _Ref(pb)
    x, y = _coords(pb)
    fields = [_phi_at(p, pb, x, y) for p in [pb["phi0"]] + ([pb["phi0_2"]] if "phi0_2" in pb else [])]
    Q = _t(np.stack(fields)).reshape(1, len(fields), ref.E, ref.n).repeat(pb["M"], 1, 1, 1)
    dW = _wiener(pb, steps)
    block = max(1, int(2e9 / (8 * ref.E * ref.n * ref.n)))
    for t in range(steps):
        if pb.get("tables") is not None:
            ref.set_fields(*pb["tables"][t % 2])
        for s in range(0, pb["M"], block):
            Q[s:s + block] = ref.step(Q[s:s + block], dW[t, s:s + block], pb["ghost"][t] if "ghost" in pb else None)
        if pb.get("reseed_every", 0) and (t + 1) % pb["reseed_every"] == 0:
            Q[:] = Q.mean(0, keepdim=True)
    return Q.mean(0).reshape(-1), (Q * Q).mean(0).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "statistics":
        _, q = _sample_values(case, seed)
        return {"mean": _t(q.mean(0)), "m2": _t((q * q).mean(0)), "pdf": None}
    if kind == "batch":
        out = []
        for pb in _instances(case, seed):
            mean, m2 = _exact_one(pb, case["steps"])
            E = int(np.prod(pb["K"]))
            out.append((mean.reshape(E, -1), m2.reshape(E, -1)))
        return out
    pb = _problem(case, seed)
    mean, m2 = _exact_one(pb, case["steps"])
    if kind == "solve":
        mean, m2 = mean.reshape(pb["K"][0], -1), m2.reshape(pb["K"][0], -1)
    return {"mean": mean, "m2": m2}
