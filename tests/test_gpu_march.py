"""The register-marching ENO2/ENO3 kernel (tile pair 6) against the FP64
oracle and, bit for bit, the scalar body at the edges of its tiles, and the
tiles chosen by default."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import (U32, compare, flip_allowance, rate_tol, rounded, step_flip_allowance,
                         to_dev)
from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PER = {3: [[True] * 3, [False] * 3, [False, False, True], [True, False, False]],
       4: [[True] * 4, [False] * 4, [False, False, True, False], [True, False, False, True]]}
# tiles that divide the axes, whose last one is moved back by one node or
# more, of one block of rows, chunks of one plane, even, odd and past the end
CASES = [([7, 14, 30], (30, 14, 7)), ([9, 15, 31], (16, 12, 2)), ([12, 8, 65], (33, 8, 1)),
         ([19, 33, 17], (17, 22, 5)), ([8, 9, 40], (20, 8, 300)),
         ([7, 9, 14, 30], (30, 14, 3)), ([8, 7, 13, 33], (17, 8, 2)), ([9, 8, 8, 41], (21, 8, 1)),
         ([10, 12, 18, 16], (16, 16, 300))]


def _spec(n, per, scheme, dyn):
    d = len(n)
    prm = {"translate": [0.7, -1.1, 0.4, 0.9][:d], "normal_speed": [1.3]}[dyn]
    s = W.problem(d, n, [-1, -1, 0, -2][:d], [1, 1.5, 2, 1][:d], per, scheme, dyn, prm, rk=3, cfl=0.75)
    s["tube"] = True
    return s


def _check(spec, tile):
    phi = rounded(W.smooth_field(spec, seed=8) + 0.2 * W.rough_field(spec, seed=9), "f32")
    g = rounded(phi + 0.05 * W.smooth_field(spec, seed=3), "f32")
    want, alpha = oracle.rate(spec, phi)
    dt = oracle.cfl_dt(spec, oracle.alpha(spec, phi), 0.75, 0.0, 10.0)
    tol = rate_tol(spec, phi, want, alpha)
    tol_step = 3 * dt * tol + 8 * U32 * np.abs(phi).max()
    P = B.Problem(spec, check_finite=True)
    if tile:
        P.set_tile(*tile, 3, 6)
        assert P.tile() == tile + (3, 6)
    assert P.tile()[4] == 6
    S = B.Problem(spec)  # the scalar body: the same operations
    S.set_tile(32, 8, 4, 3, 0)
    x = to_dev(phi, "f32")
    out, y = torch.empty_like(x), x.clone()
    P.rate(x, out)
    compare(out.double().cpu().numpy(), want, tol, flip_allowance(spec, phi, alpha), max_frac=0.05)
    P.step(x, to_dev(g, "f32"), t=0.0, dt=dt)
    S.step(y, to_dev(g, "f32"), t=0.0, dt=dt)
    assert torch.equal(x, y)
    got = x.double().cpu().numpy()
    compare(got, oracle.step(spec, phi, dt, 3, target=g), tol_step,
            step_flip_allowance(spec, phi, dt, 3, alpha, tol_step))
    assert np.all(got <= g)


@pytest.mark.parametrize("scheme", ["eno2", "eno3"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_march_tiles_match_oracle(case, scheme):
    n, tile = CASES[case]
    for i, per in enumerate(PER[len(n)]):
        _check(_spec(n, per, scheme, "translate" if i % 2 else "normal_speed"), tile)


@pytest.mark.parametrize("scheme", ["eno2", "eno3"])
def test_default_tiles_are_marches_and_match_oracle(scheme):
    for spec in (W.air3d(nx=[37, 29, 45], scheme=scheme)[0], W.car4d(n=14, scheme=scheme)[0],
                 _spec([21, 70, 26], [False] * 3, scheme, "translate")):
        spec["tube"] = True
        _check(spec, None)


def test_march_reports_nonfinite_and_refuses_what_it_does_not_cover():
    spec = _spec([9, 15, 31], [False] * 3, "eno2", "translate")
    P = B.Problem(spec, check_finite=True)
    phi = W.smooth_field(spec, seed=8)
    phi[4, 7, 15] = np.inf
    with pytest.raises(B.LspError) as e:
        P.step(to_dev(phi, "f32"), to_dev(np.full(phi.shape, 1e30), "f32"), t=0.0, dt=1e-4)
    assert e.value.status == B.LSP_ENONFINITE
    # wider than the axis, odd rows, more rows than the axis, a frame
    # of more than two values per thread
    for tile in ((32, 8, 4), (31, 7, 4), (31, 16, 4), (31, 2, 4)):
        with pytest.raises(B.LspError):
            P.set_tile(*tile, 3, 6)
    # local coefficients run the scalar local body whatever the tile
    spec["diss"] = "llf"
    L, S = B.Problem(spec), B.Problem(spec)
    L.set_tile(16, 12, 4, 3, 6)
    S.set_tile(32, 8, 4, 3, 0)
    x = to_dev(W.smooth_field(spec, seed=8), "f32")
    a, b = torch.empty_like(x), torch.empty_like(x)
    assert torch.equal(L.rate(x, a), S.rate(x, b))
