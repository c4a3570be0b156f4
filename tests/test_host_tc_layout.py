"""CPU test of the sliced GEMM's shared-memory layout (csrc/h2_tc_layout.h,
compiled for the host by tests/host/tc_layout.cpp)."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not gxx or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path_factory.mktemp("layout") / "layout.so")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-o", so,
                        os.path.join(ROOT, "tests", "host", "tc_layout.cpp"), "-I",
                        os.path.join(ROOT, "paper_2403_01566_gb300", "csrc"), "-I", cuda_inc],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return ctypes.CDLL(so)


@pytest.mark.parametrize("S", [5, 7, 8])
def test_fragment_loads_stay_in_the_slices(lib, S):
    """Every load of op(B)'s fragments lies inside op(B)'s S slices, hence
    inside the launch's shared memory whatever the tile."""
    for n in (1, 8, 9, 33, 64):
        assert lib.fragment_end(S, n) <= lib.slices_end(S)
        for m in (1, 2, 64):
            assert lib.fragment_end(S, n) <= lib.behind_b(S, m, n)
