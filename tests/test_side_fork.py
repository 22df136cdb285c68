"""Side streams are waited for however their user leaves (tests/side_fork_shim.cpp
over the library's own SideFork): a launch that fails between the fork and the
join, or any of the CUDA calls themselves.
"""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if gxx is None or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("g++ or cuda_runtime.h not found")
    out = str(tmp_path_factory.mktemp("side_fork") / "libsidefork.so")
    # (-Bsymbolic: the shim's own CUDA calls, whatever the process has loaded)
    subprocess.run([gxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-w", "-Wl,-Bsymbolic", "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_1208_6350_gb300", "csrc"), "-I", inc,
                    os.path.join(HERE, "side_fork_shim.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


@pytest.mark.parametrize("leave", [0, 1])
def test_every_forked_stream_is_waited_for(lib, leave):
    made, status = ctypes.c_int(), ctypes.c_int()
    for n in range(0, lib.sf_streams() + 1):
        assert lib.sf_run(n, leave, 0, ctypes.byref(made), ctypes.byref(status)) == 0
        assert made.value == (1 + 3 * n if n else 0)  # the fork, then a wait, a record and a wait per stream
        assert (status.value != 0) == bool(leave)
        for fail in range(1, made.value + 1):
            assert lib.sf_run(n, leave, fail, ctypes.byref(made), ctypes.byref(status)) == 0, (n, fail)
            assert status.value != 0
