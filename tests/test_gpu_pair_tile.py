"""The default WENO5 tiles on 3-D grids: valid, and the oracle's rate and step
from the shortest axes to several chunks, global and local coefficients."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import U32, compare, rate_tol, rounded, to_dev
from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [[7, 7, 7], [9, 41, 8], [41, 41, 41], [20, 9, 65], [13, 70, 23]],
                         ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("diss,varform", [("glf", False), ("llf", True)])
def test_default_weno5_tile_matches_oracle(n, diss, varform):
    spec = W.air3d(nx=n)[0]
    spec.update(tube=True, diss=diss, varform=varform)
    phi = rounded(W.smooth_field(spec, seed=8) + 0.2 * W.rough_field(spec, seed=9), "f32")
    g = rounded(phi + 0.05 * W.smooth_field(spec, seed=3), "f32")
    want, alpha = oracle.rate(spec, phi)
    P = B.Problem(spec, check_finite=True)
    x = to_dev(phi, "f32")
    out = torch.empty_like(x)
    P.rate(x, out)
    tol = rate_tol(spec, phi, want, alpha)
    compare(out.double().cpu().numpy(), want, tol)
    dt = B.lsp_cfl_dt(P.grid, P.opts, 0.0, 1e9)
    P.step(x, to_dev(g, "f32"), t=0.0, dt=dt)
    got = x.double().cpu().numpy()
    compare(got, oracle.step(spec, phi, dt, 3, target=g),
            3 * dt * tol + 8 * U32 * np.abs(phi).max())
