"""Local coefficients on tiles of the marching kernel (pair 6), whose launch
has half the z-blocks of the scalar body it falls back to in 4-D."""
import pytest
import torch

from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# 260 x 260 z-blocks of one plane; more slabs than the scalar body can launch
@pytest.mark.parametrize("n,tile,same", [([260, 260, 14, 16], (16, 14, 1), (32, 8, 2, 3, 0)),
                                         ([70000, 7, 7, 7], (7, 6, 7), (-1,))],
                         ids=["longer_chunks", "generic"])
def test_local_coefficients_on_a_march_tile_near_the_grid_limit(n, tile, same):
    spec = W.problem(4, n, [-1] * 4, [1] * 4, [False, True, False, False], "eno2", "translate",
                     [0.7, -1.1, 0.4, 0.9], rk=1, cfl=0.5)
    spec["diss"] = "llf"
    P, S = B.Problem(spec, check_finite=True), B.Problem(spec)
    P.set_tile(*tile, 3, 6)
    S.set_tile(*same)
    x = torch.rand(n, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    a, b = torch.empty_like(x), torch.empty_like(x)
    assert torch.equal(P.rate(x, a), S.rate(x, b))
