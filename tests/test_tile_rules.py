"""Default tiles of the paired WENO5 kernel (csrc/tile_rules.h, host
arithmetic)."""
import ctypes
import os
import random
import subprocess
import time

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2411_03501_gb300", "csrc")
SHIM = r"""
#include "tile_rules.h"
extern "C" void rule(const int* n, long long sms, int* out)
{
    const lsp::RuleTile t = lsp::pair_rule(n, sms), q = lsp::pair_square_tile(3, n, sms);
    out[0] = t.tb; out[1] = t.ta; out[2] = t.ch; out[3] = q.ch;
}
extern "C" int wasteful(const int* n, int tb, int ta, int ch, int threads, long long sms)
{
    return lsp::march_wasteful(n, {tb, ta, ch}, threads, sms);
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"),
                    "-o", str(d / "shim.so")], check=True)
    lib = ctypes.CDLL(str(d / "shim.so"))

    def call(n, sms=152):
        out = (ctypes.c_int * 4)()
        lib.rule((ctypes.c_int * 3)(*n), ctypes.c_longlong(sms), out)
        return tuple(out[:3]), (16, 16, out[3])
    call.lib = lib
    return call


@pytest.mark.parametrize("n,slow", [([283, 95, 74], (37, 6, 4)), ([51, 568, 172], (16, 14, 26)),
                                    ([47, 75, 400], (40, 4, 12)), ([548, 74, 14], (14, 11, 2)),
                                    ([14, 330, 336], (16, 10, 2)), ([77, 473, 64], (32, 5, 20)),
                                    ([37, 265, 157], (10, 19, 2)), ([20, 500, 500], None)])
def test_grids_where_a_fitted_tile_is_slower(rule, n, slow):
    """Timed at 7 to 30 % above the square tile: not chosen."""
    t, _ = rule(n)
    assert t != slow
    if slow is None:
        assert t[2] == 0


@pytest.mark.parametrize("n", [[41, 41, 41], [129, 129, 129], [97, 113, 85], [25, 60, 90]])
def test_grids_where_a_fitted_tile_is_faster(rule, n):
    """Timed at 10 to 40 % below the square tile."""
    assert rule(n)[0][2] > 0


def test_tiles_can_be_launched(rule):
    rng = random.Random(3)
    grids = [[7, 7, 7], [7, 7, 8], [7, 700000, 8], [7, 300000, 64], [200000, 7, 9], [7, 7, 1000000]]
    grids += [[int(7 * 100 ** rng.random()) for _ in range(3)] for _ in range(400)]
    t0 = time.perf_counter()
    for n in grids:
        (tb, ta, ch), square = rule(n)
        assert square[2] % 2 == 0 and square[2] >= 2
        if ch == 0:
            continue
        assert 8 <= tb <= min(64, n[2]) and 4 <= ta <= n[1] and 64 <= tb * ta <= 256 and ch % 2 == 0
        assert (ta + 6) * (tb + 6) <= 3 * ta * tb
        assert -(-n[1] // ta) <= 65535 and -(-n[0] // ch) <= 65535
    # chosen when a grid gets its dynamics: microseconds, whatever the axes
    assert (time.perf_counter() - t0) / len(grids) < 2e-3


@pytest.mark.parametrize("n,tile,wasteful", [([69, 14, 7, 800], (45, 6, 14, 160), True),
                                             ([7, 7, 7, 3000], (45, 6, 7, 160), True),
                                             ([7, 53, 7, 497], (46, 6, 11, 160), False),
                                             ([47, 72, 7, 169], (34, 6, 15, 128), False),
                                             ([81, 81, 81, 81], (41, 12, 27, 256), False)])
def test_march_tiles_that_compute_most_nodes_twice(rule, n, tile, wasteful):
    """Slower than the scalar kernel where timed, and the ones next to them
    that are faster."""
    assert bool(rule.lib.wasteful((ctypes.c_int * 4)(*n), *tile, ctypes.c_longlong(152))) == wasteful
