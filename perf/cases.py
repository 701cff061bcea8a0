"""The measured work: complete calls of the public API on the framework's own
workloads, from one small 2-D grid to 43 M nodes, with FP64 answers to hold
the results against.

A case names a grid, a scheme, the dynamics and how many CFL steps one call
advances.  ``prepare`` builds what a program holds before the call (the grid
handle and its workspace, the fields on the GPU), ``run`` makes the call, and
``exact`` integrates the same discrete problem in FP64 with plain torch.
Targets are unions of two discs (cylinders in higher dimensions) drawn from
the seed, as the reachability examples use them: signed distances with a kink
where the two meet.
"""
from __future__ import annotations

import math
import random

import torch
from torch.utils.checkpoint import checkpoint

from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W
from paper_2411_03501_gb300.autograd import HJTube

DEV = "cuda"
TWO_PI = 2.0 * math.pi

# bounds, periodic axes and the radius of the target of each dynamics' grid
GRIDS = {
    "normal_speed": ([-1, -1], [1, 1], [False, False], 0.3),
    "quadratic": ([-1, -1], [1, 1], [False, False], 0.3),
    "double_integrator": ([-1, -1], [1, 1], [False, False], 0.1),
    "air3d": ([-6, -10, 0], [20, 10, TWO_PI], [False, False, True], 5.0),
    "rockets": ([-64, -64, -math.pi / 2], [64, 64, math.pi / 2], [False, False, False], 1.5),
    "car4d": ([-4, -4, 0, 0], [4, 4, TWO_PI, 2], [False, False, True, False], 0.5),
}
PARAMS = {
    "normal_speed": [1.0],
    "quadratic": [],
    "double_integrator": [1.0],
    "air3d": [5.0, 5.0, 1.0, 1.0],
    "rockets": [1.0, 32.0, 1.0, 1.0],
    "car4d": [1.0, 1.0],
}


def _solve(name, dyn, n, scheme, rk, cfl, steps, dtype="f32", tube=True, diss="glf",
           varform=False, graph=False):
    c = {"kind": "solve", "dyn": dyn, "n": n, "scheme": scheme, "rk": rk, "cfl": cfl,
         "steps": steps, "dtype": dtype, "tube": tube, "diss": diss, "varform": varform,
         "graph": graph}
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the expanding 2-D front, whole: 112 stages on 10^4 nodes in one
        # graph, where launches and the chain of one node count
        _solve("front_101_f64", "normal_speed", "101x101", "eno2", 2, 0.9, 56, dtype="f64",
               tube=False, graph=True),
        # H = |p|^2/2 chooses its step from the field: one reduction and one
        # host round trip a step
        _solve("quadratic_257_f32", "quadratic", "257x193", "weno5", 3, 0.75, 12, tube=False),
        # a small pursuit game, called step range by step range
        _solve("air3d_41", "air3d", "41x41x41", "weno5", 3, 0.75, 24),
        # the pursuit game at its full size: one stretch of the horizon
        _solve("air3d_201", "air3d", "201x201x201", "weno5", 3, 0.75, 12),
        # its variational form with local dissipation on a ragged grid
        _solve("air3d_llf_varform_ragged", "air3d", "97x113x85", "weno5", 3, 0.75, 12,
               diss="llf", varform=True),
        # the 4-D car at its full size and on a ragged grid
        _solve("car4d_81", "car4d", "81x81x81x81", "eno3", 3, 0.75, 2),
        _solve("car4d_ragged", "car4d", "33x41x37x29", "eno3", 3, 0.75, 8),
        # the rockets game on the paper's grid (one of its eleven output
        # intervals, as a graph) and on fields larger than the L2 cache
        _solve("rockets_100", "rockets", "100x100x100", "eno2", 2, 0.75, 57, graph=True),
        _solve("rockets_300", "rockets", "300x300x300", "eno2", 2, 0.75, 6),
        # many problems in one call, half fronts and half games
        {"name": "batched_24", "kind": "batched", "count": 24, "scale": 1.0, "steps": 10,
         "persistent": True},
        # the gradient of a tube: forward, loss and reverse sweep
        {"name": "adjoint_129", "kind": "adjoint", "n": "129x129x129", "steps": 12, "ncheck": -1,
         "queries": 1024},
        # a target built on the device: cylinder, box, union
        {"name": "shapes_201", "kind": "shapes", "n": "201x201x201", "dtype": "f32"},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["2d", "2d", "air3d", "air3d", "air3d", "rockets", "rockets", "car4d",
                       "car4d", "batched", "adjoint", "shapes"])
    if kind == "2d":
        dyn = rng.choice(["normal_speed", "double_integrator", "quadratic"])
        n = "%dx%d" % (_log(rng, 33, 513), _log(rng, 33, 513))
        scheme, rk = rng.choice([("eno2", 2), ("eno2", 2), ("weno5", 3)])
        return _solve("", dyn, n, scheme, rk, 0.75, rng.randint(8, 64),
                      dtype=rng.choice(["f64", "f32"]), tube=dyn == "double_integrator",
                      graph=dyn != "quadratic" and rng.random() < 0.5)
    if kind == "air3d":
        n = "x".join(str(_log(rng, 25, 201)) for _ in range(3))
        return _solve("", "air3d", n, "weno5", 3, 0.75, rng.randint(4, 16),
                      diss=rng.choice(["glf", "glf", "llf"]), varform=rng.random() < 0.25,
                      graph=rng.random() < 0.25)
    if kind == "rockets":
        n = "x".join(str(_log(rng, 40, 300)) for _ in range(3))
        return _solve("", "rockets", n, "eno2", 2, 0.75, rng.randint(4, 16),
                      graph=rng.random() < 0.5)
    if kind == "car4d":
        n = "x".join(str(_log(rng, 15, 81)) for _ in range(4))
        return _solve("", "car4d", n, "eno3", 3, 0.75, rng.randint(2, 6))
    if kind == "batched":
        return {"kind": "batched", "count": 2 * rng.randint(2, 16),
                "scale": round(rng.uniform(0.3, 1.0), 3), "steps": rng.randint(4, 12),
                "persistent": rng.random() < 0.5}
    if kind == "adjoint":
        n = "x".join(str(_log(rng, 25, 129)) for _ in range(3))
        return {"kind": "adjoint", "n": n, "steps": rng.randint(3, 12),
                "ncheck": rng.choice([-1, 0]), "queries": rng.randint(16, 1024)}
    n = "x".join(str(_log(rng, 33, 257)) for _ in range(3))
    return {"kind": "shapes", "n": n, "dtype": rng.choice(["f32", "f32", "f64"])}


# ------------------------------------------------------------- the problems
def _spec(dyn, n, scheme, rk, cfl, dtype="f32", tube=True, diss="glf", varform=False,
          params=None):
    lo, hi, per, _ = GRIDS[dyn]
    n = [int(v) for v in n.split("x")] if isinstance(n, str) else n
    return W.problem(len(n), n, lo, hi, per, scheme, dyn, PARAMS[dyn] if params is None else params,
                     rk=rk, cfl=cfl, t_final=1.0, dtype=dtype, tube=tube, diss=diss,
                     varform=varform)


def _axes(spec):
    """Node coordinates of every axis, FP64, shaped to broadcast."""
    out = []
    for k in range(spec["ndim"]):
        n, lo, hi = spec["n"][k], spec["lo"][k], spec["hi"][k]
        dx = (hi - lo) / (n if spec["periodic"][k] else n - 1)
        x = lo + dx * torch.arange(n, dtype=torch.float64, device=DEV)
        out.append(x.reshape([-1 if j == k else 1 for j in range(spec["ndim"])]))
    return out


def _dx(spec):
    return [(spec["hi"][k] - spec["lo"][k]) / (spec["n"][k] - (0 if spec["periodic"][k] else 1))
            for k in range(spec["ndim"])]


def _discs(spec, rng, radius):
    """Signed distance to the union of two discs in the first two axes."""
    x = _axes(spec)
    half = [0.5 * (spec["hi"][k] - spec["lo"][k]) for k in range(2)]
    out = None
    for scale in (1.0, 0.6):
        r = radius * scale * rng.uniform(0.9, 1.1)
        c = [rng.uniform(-0.15, 0.15) * half[k] for k in range(2)]
        f = torch.sqrt((x[0] - c[0]) ** 2 + (x[1] - c[1]) ** 2) - r
        out = f if out is None else torch.minimum(out, f)
    return out.expand(spec["n"]).contiguous()


def _smooth(spec, rng, amp, modes=3):
    """Smooth field over every axis (periodic on the periodic ones)."""
    x = _axes(spec)
    out = torch.zeros(spec["n"], dtype=torch.float64, device=DEV)
    for _ in range(modes):
        term = amp * rng.uniform(0.5, 1.0)
        for k in range(spec["ndim"]):
            L = spec["hi"][k] - spec["lo"][k]
            f = rng.randint(1, 2) if spec["periodic"][k] else rng.uniform(0.3, 1.2)
            term = term * torch.sin(TWO_PI * f * (x[k] - spec["lo"][k]) / L + rng.uniform(0, TWO_PI))
        out = out + term
    return out


def _alpha(spec, prm=None):
    """Global-LF coefficients: maxima over the nodes of the bounds on |dH/dp_k|."""
    x = _axes(spec)
    p = spec["params"] if prm is None else prm
    dyn = spec["dyn"]
    if dyn == "normal_speed":
        return [abs(p[0])] * spec["ndim"]
    if dyn == "double_integrator":
        return [x[1].abs().max(), abs(p[0])]
    if dyn == "air3d":
        return [(-p[0] + p[1] * torch.cos(x[2])).abs().max() + p[2] * x[1].abs().max(),
                (p[1] * torch.sin(x[2]).abs()).max() + p[2] * x[0].abs().max(), p[2] + p[3]]
    if dyn == "car4d":
        v = x[3].abs().max()
        return [v * torch.cos(x[2]).abs().max(), v * torch.sin(x[2]).abs().max(), p[0], p[1]]
    if dyn == "rockets":
        return [p[0] * torch.cos(x[2]).abs().max() + p[2] * x[0].abs().max(),
                (p[0] * torch.sin(x[2]) + p[0] - p[1]).abs().max() + p[3] * x[0].abs().max(),
                p[2] + p[3]]
    raise ValueError(dyn)


def _cfl_dt(spec):
    return spec["cfl"] / sum(float(a) / h for a, h in zip(_alpha(spec), _dx(spec)))


def _horizon(spec, steps):
    """End time that `steps` CFL steps reach, the last one half as long."""
    if spec["dyn"] == "quadratic":  # |p| stays near 1 on a signed distance
        return 0.75 * (steps - 0.5) / sum(1.0 / h for h in _dx(spec))
    return (steps - 0.5) * _cfl_dt(spec)


def _batch(case, seed):
    rng = random.Random(seed)
    out = []
    half = case["count"] // 2
    for i in range(case["count"]):
        lo, hi = (64, 256) if i < half else (48, 128)
        # the sides are the case's, the speeds and targets the seed's
        side = max(9, int(round(case["scale"] * (lo + (hi - lo) * ((i % half) + 0.5) / half))))
        speed = rng.uniform(2.0, 6.0)
        if i < half:
            spec = _spec("normal_speed", [side, side], "weno5", 3, 0.75, params=[speed])
            radius = 0.4
        else:
            spec = _spec("air3d", [side] * 3, "weno5", 3, 0.75, params=[speed, speed, 1.0, 1.0])
            radius = 4.0
        g = _discs(spec, rng, radius).float()
        # step counts from half the case's to all of it
        steps = max(1, case["steps"] - (i * 7) % (case["steps"] // 2 + 1))
        out.append((spec, g, _horizon(spec, steps)))
    return out


def _solve_inputs(case, seed):
    spec = _spec(case["dyn"], case["n"], case["scheme"], case["rk"], case["cfl"], case["dtype"],
                 case["tube"], case["diss"], case["varform"])
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    g = _discs(spec, random.Random(seed), GRIDS[case["dyn"]][3]).to(dt)
    return spec, g, _horizon(spec, case["steps"])


def _adjoint_inputs(case, seed):
    """A tube that starts from a field crossing its target (as after a
    warm start), both with structure along every axis."""
    rng = random.Random(seed)
    spec = _spec("air3d", case["n"], "weno5", 3, 0.75)
    g = _discs(spec, rng, 5.0) + _smooth(spec, rng, 0.3)
    phi0 = g + _smooth(spec, rng, 0.3)
    q = torch.tensor([[rng.uniform(spec["lo"][k], spec["hi"][k]) for k in range(3)]
                      for _ in range(case["queries"])], dtype=torch.float32, device=DEV)
    return spec, phi0.float(), g.float(), q


def _shape_inputs(case, seed):
    rng = random.Random(seed)
    spec = _spec("air3d", case["n"], "weno5", 3, 0.75)
    return spec, {"center": [rng.uniform(-1, 1), rng.uniform(-1, 1), 0.0],
                  "radius": rng.uniform(4, 6), "lo": [rng.uniform(1, 3), -3.0, 0.0],
                  "hi": [12.0, rng.uniform(2, 4), 6.0]}


def prepare(case, seed):
    if case["kind"] == "solve":
        spec, g, t = _solve_inputs(case, seed)
        return {"kind": "solve", "P": B.Problem(spec, use_graph=case["graph"]), "phi0": g,
                "phi": torch.empty_like(g), "target": g if case["tube"] else None, "t": t}
    if case["kind"] == "batched":
        probs = _batch(case, seed)
        offs, total = [], 0
        for _, g, _ in probs:
            offs.append(total)
            total += (g.numel() + 63) // 64 * 64
        start = torch.zeros(total, dtype=torch.float32, device=DEV)
        for o, (_, g, _) in zip(offs, probs):
            start[o:o + g.numel()] = g.reshape(-1)
        work = torch.empty_like(start)
        phis = [work[o:o + g.numel()].view(g.shape) for o, (_, g, _) in zip(offs, probs)]
        return {"kind": "batched", "batch": B.Batch([p[0] for p in probs],
                                                    persistent=case["persistent"]),
                "start": start, "work": work, "phis": phis, "targets": [p[1] for p in probs],
                "t": [p[2] for p in probs]}
    if case["kind"] == "adjoint":
        spec, phi0, g, q = _adjoint_inputs(case, seed)
        return {"kind": "adjoint", "tube": HJTube(spec, case["steps"], ncheck=case["ncheck"]),
                "phi0": phi0.requires_grad_(), "target": g.requires_grad_(), "q": q,
                "params": torch.tensor(spec["params"], dtype=torch.float64, requires_grad=True)}
    spec, s = _shape_inputs(case, seed)
    grid = B.lsp_grid_create(3, spec["lo"], spec["hi"], spec["n"],
                             ["periodic" if p else "extrapolate" for p in spec["periodic"]])
    dt = torch.float64 if case["dtype"] == "f64" else torch.float32
    f = [torch.empty(spec["n"], dtype=dt, device=DEV) for _ in range(3)]
    return {"kind": "shapes", "grid": grid, "s": s, "f": f}


def run(state):
    if state["kind"] == "solve":
        # the solve works in place: the start is kept for the next call
        state["phi"].copy_(state["phi0"])
        st = state["P"].solve(state["phi"], state["target"], 0.0, state["t"])
        return {"phi": state["phi"], "steps": st["steps"]}
    if state["kind"] == "batched":
        state["work"].copy_(state["start"])
        st = state["batch"].solve(state["phis"], state["targets"], state["t"])
        return {"phi": state["phis"], "steps": [s["steps"] for s in st]}
    if state["kind"] == "adjoint":
        leaves = [state["phi0"], state["target"], state["params"]]
        for v in leaves:
            v.grad = None
        phi = state["tube"](*leaves)
        loss = state["tube"].loss(phi, state["q"])
        loss.backward()
        return {"phi": phi.detach(), "loss": loss.detach(), "grad_phi0": leaves[0].grad,
                "grad_target": leaves[1].grad, "grad_params": leaves[2].grad}
    g, s, f = state["grid"], state["s"], state["f"]
    B.lsp_shape_sphere(g, f[0], s["center"], s["radius"], ignore=(2,))
    B.lsp_shape_box(g, f[1], s["lo"], s["hi"], ignore=(2,))
    B.lsp_shape_op("union", f[0], f[1], f[2])
    return {"sphere": f[0], "box": f[1], "union": f[2]}


# --------------------------------------------------------------------- work
# operations per node and axis for both one-sided derivatives, and per node
# for the Hamiltonian
_AXIS_FLOPS = {"upwind1": 4, "eno2": 15, "eno3": 32, "weno5": 156}
_HAM_FLOPS = {"normal_speed": 6, "quadratic": 5, "double_integrator": 5, "air3d": 15, "rockets": 17,
              "car4d": 10}


def _stage_flops(spec):
    d = spec["ndim"]
    return d * (_AXIS_FLOPS[spec["scheme"]] + 5) + _HAM_FLOPS[spec["dyn"]] + 7


def work(case):
    if case["kind"] == "solve":
        spec = _spec(case["dyn"], case["n"], case["scheme"], case["rk"], case["cfl"],
                     case["dtype"], case["tube"])
        npts = math.prod(spec["n"])
        size = 8 if case["dtype"] == "f64" else 4
        return {"bytes": npts * size * (3 if case["tube"] else 2),
                "flops": npts * _stage_flops(spec) * case["steps"] * case["rk"]}
    if case["kind"] == "batched":
        b = fl = 0
        half = case["count"] // 2
        for i in range(case["count"]):
            lo, hi = (64, 256) if i < half else (48, 128)
            side = max(9, int(round(case["scale"] * (lo + (hi - lo) * ((i % half) + 0.5) / half))))
            steps = max(1, case["steps"] - (i * 7) % (case["steps"] // 2 + 1))
            dyn, d = ("normal_speed", 2) if i < half else ("air3d", 3)
            b += side ** d * 12
            fl += side ** d * steps * 3 * (d * 161 + _HAM_FLOPS[dyn] + 7)
        return {"bytes": b, "flops": fl}
    npts = math.prod(int(v) for v in case["n"].split("x"))
    if case["kind"] == "adjoint":
        # reads phi0 and the target, writes phi, the loss and two gradients;
        # the reverse of a stage counts as two forward ones
        return {"bytes": npts * 20, "flops": npts * case["steps"] * 3 * 505 * 3}
    size = 8 if case["dtype"] == "f64" else 4
    return {"bytes": npts * 5 * size, "flops": npts * 18}


# -------------------------------------------------------------------- exact
# The discrete problem in FP64 with plain torch: ghost cells, one-sided
# derivatives, Lax-Friedrichs rate, TVD-RK stages, tube.
def _ghosted(u, k, G, periodic):
    n = u.shape[k]
    if periodic:
        return torch.cat([u.narrow(k, n - G, G), u, u.narrow(k, 0, G)], k)
    j = torch.arange(1, G + 1, dtype=u.dtype, device=u.device)
    j = j.reshape([-1 if a == k else 1 for a in range(u.dim())])
    u0, u1 = u.narrow(k, 0, 1), u.narrow(k, 1, 1)
    un, um = u.narrow(k, n - 1, 1), u.narrow(k, n - 2, 1)
    return torch.cat([u0 + j.flip(k) * (u0 - u1), u, un + j * (un - um)], k)


def _pick(cond_a, cond_b, a, b):
    return torch.where(cond_a.abs() <= cond_b.abs(), a, b)


def _weno(v1, v2, v3, v4, v5):
    mx = torch.maximum(torch.maximum(torch.maximum(v1 * v1, v2 * v2),
                                     torch.maximum(v3 * v3, v4 * v4)), v5 * v5)
    eps = 1e-6 * mx + 1e-99
    s1 = 13 / 12 * (v1 - 2 * v2 + v3) ** 2 + 0.25 * (v1 - 4 * v2 + 3 * v3) ** 2 + eps
    s2 = 13 / 12 * (v2 - 2 * v3 + v4) ** 2 + 0.25 * (v2 - v4) ** 2 + eps
    s3 = 13 / 12 * (v3 - 2 * v4 + v5) ** 2 + 0.25 * (3 * v3 - 4 * v4 + v5) ** 2 + eps
    # weights scaled by eps^2, so that flat stencils stay in range
    a1, a2, a3 = 0.1 * (eps / s1) ** 2, 0.6 * (eps / s2) ** 2, 0.3 * (eps / s3) ** 2
    p1 = v1 / 3 - v2 * (7 / 6) + v3 * (11 / 6)
    p2 = -v2 / 6 + v3 * (5 / 6) + v4 / 3
    p3 = v3 / 3 + v4 * (5 / 6) - v5 / 6
    return (a1 * p1 + a2 * p2 + a3 * p3) / (a1 + a2 + a3)


def _sided(u, k, h, scheme, periodic):
    """The left and right derivatives along axis k."""
    G = 2 if scheme == "eno2" else 3
    n = u.shape[k]
    P = _ghosted(u, k, G, periodic)
    d = P.narrow(k, 1, n + 2 * G - 1) - P.narrow(k, 0, n + 2 * G - 1)

    def at(f, j):
        return f.narrow(k, j, n)

    if scheme == "weno5":
        d = d / h
        return (_weno(*(at(d, j) for j in range(5))),
                _weno(*(at(d, j) for j in range(5, 0, -1))))
    S = d.narrow(k, 1, n + 2 * G - 2) - d.narrow(k, 0, n + 2 * G - 2)  # at(S, G - 1): own node
    Sl, S0, Sr = at(S, G - 2), at(S, G - 1), at(S, G)
    pm, pp = at(d, G - 1) + 0.5 * _pick(Sl, S0, Sl, S0), at(d, G) - 0.5 * _pick(S0, Sr, S0, Sr)
    if scheme == "eno3":
        T = S.narrow(k, 1, n + 3) - S.narrow(k, 0, n + 3)
        T = [at(T, j) for j in range(4)]  # T_-2 .. T_1
        M = [_pick(T[j], T[j + 1], T[j], T[j + 1]) for j in range(3)]
        pm = pm + _pick(Sl, S0, M[0] / 3, -M[1] / 6)
        pp = pp + _pick(S0, Sr, -M[1] / 6, M[2] / 3)
    return pm / h, pp / h


def _ham(dyn, x, p, c):
    if dyn == "normal_speed":
        return c[0] * torch.sqrt(sum(q * q for q in p))
    if dyn == "quadratic":
        return 0.5 * sum(q * q for q in p)
    if dyn == "double_integrator":
        return -(p[0] * x[1] - c[0] * p[1].abs())
    s, co = torch.sin(x[2]), torch.cos(x[2])
    if dyn == "air3d":
        return -(p[0] * (-c[0] + c[1] * co) + p[1] * (c[1] * s)
                 + c[2] * (p[0] * x[1] - p[1] * x[0] - p[2]).abs() - c[3] * p[2].abs())
    if dyn == "car4d":
        return -(x[3] * (p[0] * co + p[1] * s) - c[0] * p[2].abs() - c[1] * p[3].abs())
    return -(p[0] * (c[0] * co) + p[1] * (c[0] * s + c[0] - c[1])
             + c[2] * (p[0] * x[0] - p[2]).abs() - c[3] * (p[1] * x[0] + p[2]).abs())


def _local(spec, x, c):
    if spec["dyn"] == "air3d":
        return [(-c[0] + c[1] * torch.cos(x[2])).abs() + c[2] * x[1].abs(),
                c[1] * torch.sin(x[2]).abs() + c[2] * x[0].abs(), c[2] + c[3]]
    raise ValueError(spec["dyn"])


def _rate(u, spec, alpha, prm, ranges=None):
    """L(u), or with `ranges` the largest |p| of every axis alone."""
    x, h = _axes(spec), _dx(spec)
    if spec["diss"] != "glf":
        alpha = _local(spec, x, prm)
    p, diss = [], 0.0
    for k in range(spec["ndim"]):
        pm, pp = _sided(u, k, h[k], spec["scheme"], spec["periodic"][k])
        if ranges is not None:
            ranges.append(torch.maximum(pm.abs().max(), pp.abs().max()))
            continue
        p.append(0.5 * (pm + pp))
        diss = diss + alpha[k] * 0.5 * (pp - pm)
    if ranges is not None:
        return ranges
    L = diss - _ham(spec["dyn"], x, p, prm)
    return torch.minimum(L, torch.zeros_like(L)) if spec["varform"] else L


_RK = {2: ((0.0, 1.0, 1.0), (0.5, 0.5, 0.5)),
       3: ((0.0, 1.0, 1.0), (0.75, 0.25, 0.25), (1 / 3, 2 / 3, 2 / 3))}


def _step(u, g, dt, spec, alpha, prm, call=lambda f, *a: f(*a)):
    v = u
    for cn, cs, cl in _RK[spec["rk"]]:
        a = _rate(v, spec, None, prm, []) if spec["dyn"] == "quadratic" else alpha
        new = cs * v + cl * dt * call(_rate, v, spec, a, prm)
        v = new + cn * u if cn else new
    return v if g is None else torch.where(g < v, g, v)


def _integrate(spec, u, g, t_final):
    prm = spec["params"]
    alpha = None if spec["dyn"] == "quadratic" else [float(a) for a in _alpha(spec)]
    t, steps = 0.0, 0
    while t < t_final - 1e-12 * abs(t_final):
        a = alpha if alpha is not None else [float(v) for v in _rate(u, spec, None, prm, [])]
        dt = min(spec["cfl"] / sum(v / h for v, h in zip(a, _dx(spec))), t_final - t)
        u = _step(u, g, dt, spec, alpha, prm)
        t, steps = t + dt, steps + 1
    return u, steps


def _loss(u, spec, q):
    h = _dx(spec)
    n, dV, eps = spec["n"], math.prod(h), max(h)
    total = (torch.sigmoid(-u / eps)).sum() * dV
    t = [(q[:, k].double() - spec["lo"][k]) / h[k] for k in range(spec["ndim"])]
    i0, i1, f = [], [], []
    for k in range(spec["ndim"]):
        if spec["periodic"][k]:
            b = torch.floor(t[k])
            f.append(t[k] - b)
            i0.append(b.long() % n[k])
            i1.append((b.long() + 1) % n[k])
        else:
            tk = t[k].clamp(0, n[k] - 1)
            b = torch.floor(tk).clamp(max=n[k] - 2)
            f.append(tk - b)
            i0.append(b.long())
            i1.append(b.long() + 1)
    for corner in range(1 << spec["ndim"]):
        bits = [(corner >> k) & 1 for k in range(spec["ndim"])]
        w = 1.0
        for k, b in enumerate(bits):
            w = w * (f[k] if b else 1.0 - f[k])
        total = total + (w * u[tuple(i1[k] if b else i0[k] for k, b in enumerate(bits))]).sum()
    return total


def exact(case, seed):
    if case["kind"] == "solve":
        spec, g, t = _solve_inputs(case, seed)
        u, steps = _integrate(spec, g.double(), g.double() if case["tube"] else None, t)
        return {"phi": u, "steps": steps}
    if case["kind"] == "batched":
        got = [_integrate(s, g.double(), g.double(), t) for s, g, t in _batch(case, seed)]
        return {"phi": [u for u, _ in got], "steps": [s for _, s in got]}
    if case["kind"] == "adjoint":
        spec, phi0, g, q = _adjoint_inputs(case, seed)
        leaves = [phi0.double().requires_grad_(), g.double().requires_grad_(),
                  torch.tensor(spec["params"], dtype=torch.float64, device=DEV, requires_grad=True)]
        alpha = _alpha(spec, leaves[2])
        dt = spec["cfl"] / sum(a / h for a, h in zip(alpha, _dx(spec)))
        u = leaves[0]
        for _ in range(case["steps"]):  # one stage's graph in memory at a time
            u = _step(u, leaves[1], dt, spec, alpha, leaves[2],
                      lambda f, *a: checkpoint(f, *a, use_reentrant=False))
        loss = _loss(u, spec, q)
        loss.backward()
        return {"phi": u.detach(), "loss": loss.detach(), "grad_phi0": leaves[0].grad,
                "grad_target": leaves[1].grad, "grad_params": leaves[2].grad.cpu()}
    spec, s = _shape_inputs(case, seed)
    x = _axes(spec)
    sph = torch.sqrt((x[0] - s["center"][0]) ** 2 + (x[1] - s["center"][1]) ** 2) - s["radius"]
    e = [torch.maximum(s["lo"][k] - x[k], x[k] - s["hi"][k]) for k in range(2)]
    away = torch.sqrt(e[0].clamp(min=0) ** 2 + e[1].clamp(min=0) ** 2)
    box = torch.where(away > 0, away, torch.maximum(e[0], e[1]))
    sph, box = (v.expand(spec["n"]).contiguous() for v in (sph, box))
    return {"sphere": sph, "box": box, "union": torch.minimum(sph, box)}
