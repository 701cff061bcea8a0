"""Stage launches that start before the previous stage has finished: a solve
enqueued back to back, and its graph, give the bits of single steps with the
device idle between them, on every kernel launched that way and from one CTA
to several waves."""
import pytest
import torch

from gpu_helpers import rounded, to_dev
from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["plane64", "plane32", "march3", "march4", "pair", "pair_waves"])
def test_back_to_back_stages_equal_synchronised_steps(kind):
    if kind.startswith("plane"):
        spec = W.problem(2, [101, 97] if kind == "plane64" else [9, 13], [-1, -1], [1, 1], [False, True],
                         "weno5", "normal_speed", [1.0], rk=3, cfl=0.75,
                         dtype="f64" if kind == "plane64" else "f32")
    elif kind == "march3":
        spec = W.problem(3, [33, 40, 61], [-1, -1, -1], [1, 1, 1], [False, False, True], "eno2",
                         "normal_speed", [1.0], rk=2, cfl=0.75)
    elif kind == "march4":
        spec = W.car4d(n=17)[0]
    else:
        spec = W.air3d(nx=[21, 23, 26] if kind == "pair" else [80, 90, 70])[0]
    spec["tube"] = True
    phi = rounded(W.smooth_field(spec, seed=8), spec["dtype"])
    g = to_dev(rounded(phi + 0.05 * W.smooth_field(spec, seed=3), spec["dtype"]), spec["dtype"])
    steps = 25
    P = B.Problem(spec)
    dt = B.lsp_cfl_dt(P.grid, P.opts, 0.0, 1e9)
    ref = to_dev(phi, spec["dtype"])
    t, t_final = 0.0, (steps - 0.5) * dt
    for _ in range(steps):
        h = min(dt, t_final - t)
        P.step(ref, g, t=t, dt=h)
        torch.cuda.synchronize()
        t += h
    for graph in (False, True):
        Q = B.Problem(spec, use_graph=graph)
        for _ in range(3):
            x = to_dev(phi, spec["dtype"])
            assert Q.solve(x, g, 0.0, t_final)["steps"] == steps
            torch.cuda.synchronize()
            assert torch.equal(x, ref)
