"""Solves whose step the device chooses from the field (H = |p|^2/2) against
the oracle: step counts and stats from no step to several batches of enqueued
steps, every RK order, dimension and stage kernel, and the call after one."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import U32, rounded, to_dev
from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _spec(n, scheme, rk, dtype, tube=False):
    d = len(n)
    s = W.problem(d, n, [-1] * d, [1] * d, [False] * (d - 1) + [True], scheme, "quadratic", [], rk=rk,
                  cfl=0.5, t_final=0.3, dtype=dtype)
    s["tube"] = tube
    return s


def _run(spec, phi, t, g=None, P=None):
    P = P or B.Problem(spec, check_finite=True)
    x = to_dev(phi, spec["dtype"])
    st = P.solve(x, None if g is None else to_dev(g, spec["dtype"]), 0.0, t)
    return x.double().cpu().numpy(), st, P


@pytest.mark.parametrize("n,rk,scheme,tube", [([41], 1, "upwind1", True), ([33, 29], 3, "weno5", False),
                                              ([33, 29], 1, "eno3", True), ([15, 17, 13], 2, "eno2", True),
                                              ([9, 8, 9, 7], 3, "eno3", False)])
def test_device_steps_match_oracle(n, rk, scheme, tube):
    spec = _spec(n, scheme, rk, "f64", tube)
    phi = rounded(W.smooth_field(spec, seed=8), "f64")
    g = rounded(phi + 0.05 * W.smooth_field(spec, seed=3), "f64") if tube else None
    _, probe = oracle.solve(spec, phi, 1.0, rk, 0.5, target=g, max_steps=1)
    P = None
    # no step, a shortened first one, one and a half, and more than a batch
    for t in (0.0, 0.4 * probe["dt_max"], 1.5 * probe["dt_max"], 40.3 * probe["dt_max"]):
        want, so = oracle.solve(spec, phi, t, rk, 0.5, target=g)
        got, st, P = _run(spec, phi, t, g, P)
        assert st["steps"] == so["steps"] and st["stages"] == rk * so["steps"]
        assert np.abs(got - want).max() <= 1e-9 * np.abs(want).max()
        if so["steps"]:
            for k in ("dt_min", "dt_max", "t_end"):
                assert abs(st[k] - so[k]) <= 1e-9 * abs(so[k]), k


@pytest.mark.parametrize("n,scheme,rk", [([21, 26, 33], "eno2", 2), ([21, 26, 33], "weno5", 3),
                                         ([12, 12, 12, 12], "eno3", 3), ([97, 61], "weno5", 3)])
def test_device_steps_on_every_fp32_kernel(n, scheme, rk):
    """FP32 solves on the tiled kernels: the same step count as FP64 on the
    GPU, and fields apart by rounding.  A smooth field: each step adds at most
    the rounding of its differences, 16 u max|phi| sum_k alpha_k dt / dx_k
    (= 16 u max|phi| cfl), and 8 u max|phi| for the combination per stage."""
    phi = rounded(W.smooth_field(_spec(n, scheme, rk, "f32"), seed=8), "f32")
    t = 0.02
    a, sa, _ = _run(_spec(n, scheme, rk, "f32"), phi, t)
    b, sb, _ = _run(_spec(n, scheme, rk, "f64"), phi, t)
    assert sa["steps"] == sb["steps"] > 1
    if scheme == "weno5":
        assert np.abs(a - b).max() <= sa["stages"] * 8 * (16 * 0.5 + 8) * U32 * np.abs(phi).max()
    assert np.isfinite(a).all()


def test_nonfinite_field_ends_the_solve():
    spec = _spec([33, 29], "eno2", 2, "f32")
    phi = W.smooth_field(spec, seed=8)
    phi[5, 5] = np.nan
    with pytest.raises(B.LspError) as e:
        _run(spec, phi, 0.1)
    assert e.value.status == B.LSP_ENONFINITE
