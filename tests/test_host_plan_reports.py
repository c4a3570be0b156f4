"""CPU test: a product's replays report its error flag whether or not it has
adaptive ranks; matrix-vector plans have nothing to report."""
import ctypes
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2403_01566_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not gxx or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    so = str(tmp_path_factory.mktemp("reports") / "reports.so")
    r = subprocess.run([gxx, "-O1", "-std=c++17", "-shared", "-fPIC", "-o", so,
                        os.path.join(ROOT, "tests", "host", "plan_reports.cpp"),
                        os.path.join(CSRC, "h2_plan.cpp"), os.path.join(CSRC, "h2_build.cpp"),
                        "-I", os.path.join(ROOT, "include"), "-I", cuda_inc], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    return ctypes.CDLL(so)


def test_product_without_ranks_reports(lib):
    reports = ctypes.c_int()
    assert lib.product_ranks(ctypes.byref(reports)) == 0
    assert reports.value
    assert not lib.matvec_reports()
