"""CPU test: a Jacobi SVD job goes only to CTAs that hold its columns."""
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
    so = str(tmp_path_factory.mktemp("svd") / "svd.so")
    r = subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-o", so,
                        os.path.join(ROOT, "tests", "host", "svd_jobs.cpp"),
                        "-I", os.path.join(ROOT, "include"), "-I", cuda_inc], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return ctypes.CDLL(so)


def test_every_column_has_a_thread_and_a_row_warp_is_left(lib):
    for threads in (128, 256):
        for cols in range(1, 257):
            if lib.cta_takes(cols, threads):
                assert threads // cols >= 1  # segments of the column norms
                assert threads // 32 - (cols + 63) // 64 >= 1
    assert all(lib.cta_takes(c, 256) for c in range(1, 257))  # the largest SVD there is


def test_small_jobs_fit_their_ctas(lib):
    for rows in range(1, 257):
        for cols in range(1, 257):
            if lib.small_job(rows, cols):
                assert lib.cta_takes(cols, 128)
    assert lib.small_job(64, 64) and not lib.small_job(8, 129)
