"""Tiles of the register-marching ENO kernel (pair 6) on the host: what
lsp_get_tile reports can be set on another handle of the same grid."""
import random

import pytest

from paper_2411_03501_gb300 import binding as B


@pytest.fixture(scope="module", autouse=True)
def lib():
    from paper_2411_03501_gb300 import build
    build.build()
    return B.load()


def _grid(n):
    d = len(n)
    g = B.lsp_grid_create(d, [0] * d, [1] * d, n, ["extrapolate"] * d)
    B.lsp_set_dynamics(g, "quadratic", [])  # no device work
    return g


@pytest.mark.parametrize("scheme", ["eno2", "eno3"])
def test_default_tiles_can_be_set(scheme):
    o = B.make_opts(rk_order=2, scheme=scheme, dtype="f32")
    rng = random.Random(4)
    grids = [[7, 7, 7], [41, 41, 41], [57, 43, 211], [250, 41, 60], [7, 7, 7, 7], [9, 12, 20, 31]]
    grids += [[int(7 * 40 ** rng.random()) for _ in range(d)] for d in [3] * 150 + [4] * 20]
    marches = 0
    for n in grids:
        t = B.lsp_get_tile(_grid(n), o)
        marches += t[4] == 6
        g = _grid(n)
        B.lsp_set_tile(g, *t)
        assert B.lsp_get_tile(g, o) == t, n
    assert marches > len(grids) // 2


def test_a_tile_of_one_scheme_runs_generic_on_the_other():
    """41 x 6: the 2-wide frame fits two values per thread, the 3-wide not."""
    g = _grid([41, 41, 41])
    B.lsp_set_tile(g, 41, 6, 6, 3, 6)
    assert B.lsp_get_tile(g, B.make_opts(scheme="eno2", dtype="f32")) == (41, 6, 6, 3, 6)
    assert B.lsp_get_tile(g, B.make_opts(scheme="eno3", dtype="f32")) == (-1,) * 5
