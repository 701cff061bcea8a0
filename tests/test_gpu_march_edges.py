"""Forms of the marching ENO kernel (pair 6) beyond its usual launches give
the scalar body's bits: a tile above 48 KB of shared memory, and the ordinary
launch that 4-D grids of many waves get."""
import pytest
import torch

from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", ["eno2", "eno3"])
@pytest.mark.parametrize("n,tile", [([8, 7, 60, 9], (9, 56, 4)), ([20, 21, 60, 61], (31, 16, 1))],
                         ids=["64_kb", "many_waves"])
def test_march_forms_equal_the_scalar_body(n, tile, scheme):
    spec = W.problem(4, n, [-1] * 4, [1] * 4, [False, True, False, True], scheme, "translate",
                     [0.7, -1.1, 0.4, 0.9], rk=3, cfl=0.5)
    spec["tube"] = True
    P, S = B.Problem(spec, check_finite=True), B.Problem(spec)
    P.set_tile(*tile, 3, 6)
    assert P.tile() == tile + (3, 6)
    S.set_tile(32, 8, 4, 3, 0)
    x = torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    g = x + 0.1 * torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    y = x.clone()
    dt = B.lsp_cfl_dt(P.grid, P.opts, 0.0, 1e9)
    assert P.solve(x, g, 0.0, 1.5 * dt)["steps"] == S.solve(y, g, 0.0, 1.5 * dt)["steps"] == 2
    assert torch.equal(x, y)


@pytest.mark.parametrize("spec", [W.rockets(n=27)[0], W.air3d(nx=[37, 29, 45], scheme="eno3")[0], W.car4d(n=15)[0]],
                         ids=["rockets", "air3d", "car4d"])
def test_march_with_a_heading_equals_the_scalar_body(spec):
    P, S = B.Problem(spec), B.Problem(spec)
    assert P.tile()[4] == 6
    S.set_tile(32, 8, 4, 3, 0)
    x = torch.rand(spec["n"], device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    y, g = x.clone(), x + 0.05
    dt = B.lsp_cfl_dt(P.grid, P.opts, 0.0, 1e9)
    P.solve(x, g, 0.0, 3.5 * dt)
    S.solve(y, g, 0.0, 3.5 * dt)
    assert torch.equal(x, y)
