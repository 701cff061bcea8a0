"""Block size of the 2-D kernels (csrc/launch.h): small grids are spread over
every SM, large ones get full blocks whatever the remainder."""
import ctypes
import os
import random
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2411_03501_gb300", "csrc")
SHIM = '#include "launch.h"\nextern "C" int block(long long n, long long s) { return lsp::plane_block(n, s); }\n'


@pytest.fixture(scope="module")
def block(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME") or os.path.dirname(os.path.dirname(
        os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    d = tmp_path_factory.mktemp("block")
    (d / "shim.cpp").write_text(SHIM)
    # the device queries of launch.h's inline functions are never called
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, "-I", cuda + "/include",
                    str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    f = ctypes.CDLL(str(d / "shim.so"), mode=os.RTLD_LAZY).block
    f.argtypes = [ctypes.c_longlong, ctypes.c_longlong]
    return f


def test_small_grids_use_every_sm(block):
    assert block(49, 152) == 64
    assert block(101 * 101, 152) == 96
    assert block(257 * 193, 152) == 192
    assert block(513 * 401, 152) == 128


def test_block_is_a_near_best_split_and_full_on_large_grids(block):
    rng = random.Random(1)
    for _ in range(300):
        n = int(49 * (2**31 / 49) ** rng.random())
        t = block(n, 152)
        assert t % 32 == 0 and 64 <= t <= 256
        busiest = {s: -(-(-(-n // s)) // 152) * s for s in range(64, 257, 32)}
        assert busiest[t] * 99 <= min(busiest.values()) * 100
    for n in (4096 * 4096, 4097 * 4095, 8192 * 8192, 20011 * 20011):
        assert block(n, 152) == 256
