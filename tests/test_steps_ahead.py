"""How many device-chosen steps are enqueued before the next read-back
(csrc/lsp_internal.h, host arithmetic)."""
import ctypes
import math
import os
import shutil
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2411_03501_gb300", "csrc")


def test_no_idle_step_where_the_last_length_fits(tmp_path):
    cuda = os.environ.get("CUDA_HOME") or os.path.dirname(os.path.dirname(
        os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    (tmp_path / "shim.cpp").write_text('#include "lsp_internal.h"\n'
                                       'extern "C" int ahead(double left) { return lsp::steps_ahead(left); }\n')
    subprocess.run(["g++", "-std=c++17", "-O2", "-shared", "-fPIC", "-I", CSRC, "-I", cuda + "/include",
                    str(tmp_path / "shim.cpp"), "-o", str(tmp_path / "shim.so")], check=True)
    f = ctypes.CDLL(str(tmp_path / "shim.so"), mode=os.RTLD_LAZY).ahead
    f.argtypes = [ctypes.c_double]
    # one shortened step left: one step, not two
    assert [f(x) for x in (1e-9, 0.3, 0.96)] == [1, 1, 1]
    assert [f(x) for x in (1.0, 1.5, 1.9, 10.5)] == [2, 2, 2, 11]
    for k in range(1, 4000):
        x = k / 8.0
        assert min(256, math.ceil(x)) <= f(x) <= min(256, math.ceil(x) + math.ceil(x / 32))
    assert f(1e300) == f(math.inf) == 256
    assert f(math.nan) == f(-1.0) == 1
