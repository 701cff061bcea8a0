"""2-D WENO5 on rough fields of any magnitude: the weights neither overflow
nor vanish."""
import numpy as np
import pytest
import torch

import oracle
from gpu_helpers import compare, rate_tol, rounded, to_dev
from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,scales", [("f32", (1.0, 1e6, 3e8, 1e9, 1e12, 1e15)),
                                          ("f64", (1e-40, 1e-6, 1e9, 1e30, 1e60))])
def test_rough_fields_of_any_magnitude(dtype, scales):
    spec = W.problem(2, [61, 67], [-1, -1], [1, 1], [False, True], "weno5", "normal_speed", [1.0],
                     dtype=dtype)
    rough = W.smooth_field(spec, seed=8) + 10 * W.rough_field(spec, seed=9)
    for s in scales:
        phi = rounded(s * rough, dtype)
        want, alpha = oracle.rate(spec, phi)
        x = to_dev(phi, dtype)
        out = torch.empty_like(x)
        B.Problem(spec, check_finite=True).rate(x, out)
        got = out.double().cpu().numpy()
        assert np.isfinite(got).all(), s
        compare(got, want, rate_tol(spec, phi, want, alpha))
