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
    ptr = np.ctypeslib.ndpointer
    lib.reciprocals.argtypes = [ptr(np.float64), ctypes.c_int, ptr(np.float64), ptr(np.float64)]
    lib.cosines.argtypes = [ptr(np.float32), ctypes.c_int, ptr(np.float64), ptr(np.float64)]
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


# A seed is off by at most 2 units of FP32 (the functions) and 2^-23 (the
# truncated operand), delta < 2^-21; a step of third order leaves 2.5 delta^3 <
# 2^-61, and its FP64 roundings less than one unit of 2^-53 beside that of the
# result: 2^-52.
BOUND = 2.0 ** -52


def _error(got, want):
    """Largest relative error against an extended-precision value."""
    return float(np.max(np.abs(got.astype(np.longdouble) / want - 1)))


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 63, reason="needs an extended precision")
@pytest.mark.parametrize("ulps", [-2, -1, 0, 1, 2])
def test_reciprocals_and_cosines(lib, ulps):
    lib.set_seed_ulps(ulps)
    try:
        rng = np.random.default_rng(6)
        # every exponent; the ends of an FP32 and an FP64 fraction; subnormal numbers (the library functions')
        m = np.concatenate([1.0 + rng.random(6), [1.0, 1.0 + 2.0 ** -52, 1.0 + 2.0 ** -23, 1.5, 2.0 - 2.0 ** -23,
                                                  2.0 - 2.0 ** -52]])
        v = np.concatenate([np.ldexp(m, e) for e in range(-1022, 1024)] + [np.ldexp(m, -1030)])
        rsq, rec = np.empty_like(v), np.empty_like(v)
        lib.reciprocals(v, len(v), rsq, rec)
        vl = v.astype(np.longdouble)
        assert _error(rsq, 1 / np.sqrt(vl)) <= BOUND
        normal = (v < 2.0 ** 1022) & (v > 2.0 ** -1022)  # (1 / v normal and finite)
        assert _error(rec[normal], (1 / vl)[normal]) <= BOUND
        with np.errstate(over="ignore"):
            assert np.array_equal(rec[~normal], 1.0 / v[~normal])
        t = np.concatenate([rng.uniform(-1, 1, 4000), 2.0 ** -rng.uniform(0, 40, 2000), [0.0, 1.0, -1.0]])
        t = t.astype(np.float32)
        q, c = np.empty(len(t)), np.empty(len(t))
        lib.cosines(t, len(t), q, c)
        assert _error(c, 1 / np.sqrt(q.astype(np.longdouble))) <= BOUND
    finally:
        lib.set_seed_ulps(0)
