"""2-D stages on grids of more nodes than one pass of the FP64 kernel's blocks
has threads (a grid-stride loop): the same bits as the same nodes get on a
small grid."""
import pytest
import torch

from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("scheme", ["upwind1", "eno2", "eno3", "weno5"])
def test_many_periods_equal_one(scheme, dtype):
    """A field of 40 x 41 equal periods on periodic axes: every period has the
    rate of one period alone (translation: no coordinate enters)."""
    n, reps = [37, 29], [40, 41]
    t = torch.float64 if dtype == "f64" else torch.float32
    one = torch.rand(n, device="cuda", dtype=t, generator=torch.Generator("cuda").manual_seed(4))
    many = one.repeat(reps).contiguous()
    rates = []
    for phi, m in ((one, [1, 1]), (many, reps)):
        spec = W.problem(2, [a * b for a, b in zip(n, m)], [0, 0], [37.0 * m[0], 29.0 * m[1]],
                         [True, True], scheme, "translate", [0.7, -1.1], dtype=dtype)
        out = torch.empty_like(phi)
        rates.append(B.Problem(spec, check_finite=True).rate(phi, out))
    assert many.numel() > 16 * 152 * 256 * 2
    assert torch.equal(rates[0].repeat(reps), rates[1])
