"""CPU test of the scalar pieces of the factorisation kernels
(csrc/h2_scalar.cuh, compiled for the host by tests/host/kernel_scalars.cpp)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not gxx or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path_factory.mktemp("scalars") / "scalars.so")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-o", so,
                        os.path.join(ROOT, "tests", "host", "kernel_scalars.cpp"), "-I",
                        os.path.join(ROOT, "paper_2403_01566_gb300", "csrc"), "-I", cuda_inc],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    lib = ctypes.CDLL(so)
    lib.threshold.restype = ctypes.c_float
    lib.threshold.argtypes = [ctypes.c_double, ctypes.c_double]
    lib.pair_tan.argtypes = [ctypes.c_double, ctypes.c_double, ctypes.c_float, ctypes.POINTER(ctypes.c_float)]
    lib.pair_tan.restype = None
    return lib


def test_lanes_of_a_jacobi_pair_agree(lib):
    """Two lanes hold a pair with its columns exchanged; next to the threshold,
    too, they must rotate by the same angle or both not rotate."""
    rng = np.random.default_rng(5)
    t = (ctypes.c_float * 2)()
    rotated = 0
    for na, nb in np.exp2(rng.uniform(-30.0, 50.0, (2000, 2))):
        thr = np.float32(lib.threshold(na, nb))
        for ulps in (-2, -1, 0, 1, 2):
            g = np.uint32(int(thr.view(np.uint32)) + ulps).view(np.float32)
            lib.pair_tan(na, nb, g, t)
            assert t[0] == t[1], (na, nb, ulps)
            rotated += t[0] != 0.0
    assert 0 < rotated < 10000
