"""Implicit surfaces on fields large enough for the kernels' 16-byte form and
for several rounds of their loops, at both alignments: the oracle's values, and
the same bits at either alignment; set operations bit for bit."""
import numpy as np
import pytest
import torch

from oracle import shapes as S
from paper_2411_03501_gb300 import binding as B
from paper_2411_03501_gb300 import workloads as W

pytestmark = pytest.mark.gpu


# more than 16 blocks of 256 threads with 4 nodes each per SM; rows shorter
# than two threads' nodes; a length that leaves a remainder
@pytest.mark.parametrize("n", [[1701, 1603], [300, 301, 7], [31, 33, 35, 13]],
                         ids=lambda n: "x".join(map(str, n)))
@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_large_fields_at_both_alignments(n, dtype):
    d = len(n)
    spec = W.problem(d, n, [-1, -2, 0, -1][:d], [1, 1, 2, 3][:d], [False] * d, "eno2", "normal_speed", [1.0])
    g = B.lsp_grid_create(d, spec["lo"], spec["hi"], n, ["extrapolate"] * d)
    size = int(np.prod(n))

    def field(off):
        return torch.zeros(size + 4, dtype=dtype, device="cuda")[off:off + size].view(n)

    c, lo, hi = [0.3, -0.4, 1.0, 0.5][:d], [-0.5, -1.0, 0.2, 0.0][:d], [0.4, 0.3, 1.5, 1.0][:d]
    w, nrm = [1.0, -0.5, 2.0, 0.25][:d], [1.0, 2.0, -0.5, 0.3][:d]
    scale = np.sqrt(d) * 5.0 + 2.0  # distances, coordinates, centre, radius
    cases = [(lambda o: B.lsp_shape_sphere(g, o, c, 1.7), S.sphere(spec, c, 1.7), scale),
             (lambda o: B.lsp_shape_sphere(g, o, c, 1.2, ignore=(d - 1,)), S.sphere(spec, c, 1.2, ignore=(d - 1,)), scale),
             (lambda o: B.lsp_shape_box(g, o, lo, hi, ignore=(0,)), S.box(spec, lo, hi, ignore=(0,)), scale),
             (lambda o: B.lsp_shape_quadric(g, o, c, w, 0.7), S.quadric(spec, c, w, 0.7), 2.0 * scale ** 2),
             (lambda o: B.lsp_shape_halfspace(g, o, nrm, c), S.halfspace(spec, nrm, c), scale)]
    tol = 1e-12 if dtype == torch.float64 else 32 * 2.0 ** -24
    kept = []
    for make, want, s in cases:
        a, b = field(0), field(1)
        make(a)
        make(b)
        assert np.abs(a.double().cpu().numpy() - want).max() <= tol * s
        assert torch.equal(a, b)
        kept.append((a, b))
    (a0, b0), (a1, b1) = kept[0], kept[2]
    for op, want in (("union", torch.minimum(a0, a1)), ("intersect", torch.maximum(a0, a1)),
                     ("complement", -a0), ("difference", torch.maximum(a0, -a1))):
        for x, y, off in ((a0, a1, 0), (b0, b1, 1), (a0, b1, 0)):
            out = field(off)
            B.lsp_shape_op(op, x, y, out)
            assert torch.equal(out, want), op
