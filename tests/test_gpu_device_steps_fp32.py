"""FP32 solves whose step the device chooses (H = |p|^2/2) against single steps
of the same field, bit for bit, on every kernel that reads the step from the
control block and skips the stages enqueued past the last one."""
import pytest
import torch

from gpu_helpers import rounded, to_dev
from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# the default kernel of each grid and scheme, the scalar body, the face-shared
# runs, paired planes, the generic kernel
CASES = [([97, 61], "weno5", 3, None), ([53], "eno3", 1, None),
         ([21, 26, 33], "eno2", 2, None), ([21, 26, 33], "eno3", 1, None), ([21, 26, 33], "weno5", 3, None),
         ([12, 13, 12, 14], "eno3", 3, None), ([12, 13, 12, 14], "weno5", 2, None),
         ([21, 26, 33], "eno3", 3, (32, 8, 4, 3, 0)), ([21, 26, 33], "eno2", 3, (16, 8, 5, 3, 3)),
         ([21, 26, 33], "eno2", 2, (32, 8, 4, 3, 1)), ([12, 13, 12, 14], "eno2", 2, (-1,))]


def _spec(n, scheme, rk):
    d = len(n)
    s = W.problem(d, n, [-1] * d, [1] * d, [False] * (d - 1) + [True], scheme, "quadratic", [], rk=rk, cfl=0.5)
    s["tube"] = True
    return s


@pytest.mark.parametrize("n,scheme,rk,tile", CASES)
@pytest.mark.parametrize("steps", [1, 2, 9])
def test_solve_equals_single_steps(n, scheme, rk, tile, steps):
    spec = _spec(n, scheme, rk)
    P = B.Problem(spec, check_finite=True)
    if tile:
        P.set_tile(*tile)
    phi = rounded(W.smooth_field(spec, seed=8), "f32")
    g = to_dev(rounded(phi + 0.05 * W.smooth_field(spec, seed=3), "f32"), "f32")
    x, y, t = to_dev(phi, "f32"), to_dev(phi, "f32"), 0.0
    for _ in range(steps):
        t += P.step(x, g, t=t, dt=0.0)
    st = P.solve(y, g, 0.0, t)
    assert st["steps"] == steps and abs(st["t_end"] - t) <= 1e-15 * t
    assert torch.equal(x, y)


@pytest.mark.parametrize("n,scheme,rk", [([21, 26, 33], "eno2", 2), ([21, 26, 33], "eno3", 3),
                                         ([12, 13, 12, 14], "eno3", 3)])
def test_march_solves_equal_the_scalar_body(n, scheme, rk):
    spec = _spec(n, scheme, rk)
    P, S = B.Problem(spec), B.Problem(spec)
    assert P.tile()[4] == 6
    S.set_tile(32, 8, 4, 3, 0)
    phi = rounded(W.smooth_field(spec, seed=8), "f32")
    g = to_dev(rounded(phi + 0.05 * W.smooth_field(spec, seed=3), "f32"), "f32")
    x, y = to_dev(phi, "f32"), to_dev(phi, "f32")
    assert P.solve(x, g, 0.0, 0.02)["steps"] == S.solve(y, g, 0.0, 0.02)["steps"] > 1
    assert torch.equal(x, y)
