"""The 2-D stage kernel against the FP64 oracle at the edges of its range:
axes as short as the stencil, node counts around a block and around one block
per SM, ghosts of both kinds, flat fields, and the costate range."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import compare, flip_allowance, rate_tol, rounded, to_dev
from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [[7, 7], [7, 40], [33, 8], [64, 152], [61, 131], [257, 193]]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("scheme", ["upwind1", "eno2", "eno3", "weno5"])
@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_plane_rate_matches_oracle(n, scheme, dtype):
    for per, dyn, prm in (([True, False], "quadratic", []), ([False, True], "translate", [0.7, -1.1]),
                          ([False, False], "normal_speed", [1.3])):
        spec = W.problem(2, n, [-1, -0.5], [1, 1.5], per, scheme, dyn, prm, dtype=dtype)
        phi = rounded(W.smooth_field(spec, seed=8) + 0.2 * W.rough_field(spec, seed=9), dtype)
        phi[: n[0] // 3] = phi[0, 0]  # a flat part: every indicator zero
        want, alpha = oracle.rate(spec, phi)
        x = to_dev(phi, dtype)
        out = torch.empty_like(x)
        B.Problem(spec, check_finite=True).rate(x, out)
        compare(out.double().cpu().numpy(), want, rate_tol(spec, phi, want, alpha),
                flip_allowance(spec, phi, alpha))
