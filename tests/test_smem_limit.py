"""The shared-memory limit of a kernel is raised on the device of each launch
(csrc/launch.h with a stand-in for the runtime: one machine may have one
device)."""
import ctypes
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2411_03501_gb300", "csrc")
SHIM = r"""
#include "launch.h"
static int device = 0, limit[2] = {48 * 1024, 48 * 1024};
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int v)
{
    limit[device] = v;
    return v <= 227 * 1024 ? cudaSuccess : cudaErrorInvalidValue;
}
static void kernel(int) {}
// the launcher's check, then what the launch itself would answer
extern "C" int launch_on(int dev, int smem, int most)
{
    device = dev;
    if (const cudaError_t e = lsp::allow_smem(kernel, smem, most)) return e;
    return smem <= limit[dev] ? cudaSuccess : cudaErrorInvalidValue;
}
extern "C" int limit_of(int dev) { return limit[dev]; }
"""


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    cuda = os.environ.get("CUDA_HOME") or os.path.dirname(os.path.dirname(
        os.path.realpath(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc")))
    d = tmp_path_factory.mktemp("smem")
    (d / "shim.cpp").write_text(SHIM)
    # its own stand-in, whatever runtime the process has loaded
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I", CSRC, "-I", cuda + "/include",
                    str(d / "shim.cpp"), "-o", str(d / "shim.so")], check=True)
    return ctypes.CDLL(str(d / "shim.so"))


def test_every_device_gets_the_limit(shim):
    for dev in (0, 1, 0, 1):
        assert shim.launch_on(dev, 60 * 1024, 200 * 1024) == 0
        assert shim.limit_of(dev) == 200 * 1024
        assert shim.launch_on(dev, 50 * 1024, 200 * 1024) == 0  # a smaller launch lowers nothing
        assert shim.limit_of(dev) == 200 * 1024
    assert shim.launch_on(0, 240 * 1024, 240 * 1024) != 0


def test_no_launcher_keeps_the_limit_for_the_process():
    """Every launcher that raises the limit does so through allow_smem or at
    each launch, never once in a static initialiser."""
    for f in os.listdir(CSRC):
        src = open(os.path.join(CSRC, f)).read()
        for i in [i for i in range(len(src)) if src.startswith("cudaFuncSetAttribute(", i)]:
            before = src[:i]
            start = max(before.rfind(";"), before.rfind("{"))
            assert "static" not in src[start:i], f
