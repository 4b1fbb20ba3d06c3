"""The sums of the cached-factor x-update (csrc/compsum.h) on the CPU: as good as a
float64 sum of the same float32 products, where a float32 sum of a few loses bits;
and the x-update uses them for every width."""
import ctypes as C
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2304_14568_gb300", "csrc")


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("needs g++")
    out = str(tmp_path_factory.mktemp("compsum") / "libcompsum_shim.so")
    subprocess.run([cxx, "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(HERE, "compsum_shim.cpp"), "-o", out], check=True)
    L = C.CDLL(out)
    L.shim_compsum.restype = C.c_double
    L.shim_compsum.argtypes = [np.ctypeslib.ndpointer(np.float32, flags="C"), C.c_int]
    L.shim_compsum_parts.restype = C.c_double
    L.shim_compsum_parts.argtypes = [np.ctypeslib.ndpointer(np.float32, flags="C"), C.c_int, C.c_int]
    return L


@pytest.mark.parametrize("n", [1, 3, 8, 40, 157, 1000])
@pytest.mark.parametrize("spread", [0.0, 3.0, 8.0])
def test_as_good_as_a_float64_sum(shim, n, spread):
    rng = np.random.default_rng(n)
    worst, worst32 = 0.0, 0.0
    for _ in range(50):
        p = (rng.normal(size=n) * np.exp(spread * rng.normal(size=n))).astype(np.float32)
        exact, mag = float(np.sum(p.astype(np.longdouble))), float(np.sum(np.abs(p).astype(np.float64)))
        worst = max(worst, abs(shim.shim_compsum(p, n) - exact) / mag)
        worst32 = max(worst32, abs(float(np.add.accumulate(p)[-1]) - exact) / mag)
    # every addition's error is kept in c (rounded itself): n^2 eps^2 of the sum's size
    assert worst <= 2.0 ** -50 + (n * 2.0 ** -24) ** 2
    if n >= 8 and spread == 0.0:
        assert worst < 2.0 ** -36 < worst32


@pytest.mark.parametrize("n", [1, 40, 157, 1000])
@pytest.mark.parametrize("parts", [2, 32, 64])
def test_sums_added_up_are_as_good(shim, n, parts):
    rng = np.random.default_rng(n)
    for _ in range(20):
        p = rng.normal(size=n).astype(np.float32)
        exact, mag = float(np.sum(p.astype(np.longdouble))), float(np.sum(np.abs(p).astype(np.float64)))
        assert abs(shim.shim_compsum_parts(p, n, parts) - exact) <= (2.0 ** -50 + (n * 2.0 ** -24) ** 2) * mag


def test_the_x_update_sums_every_product_this_way():
    src = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "solver.cu")).read())
    at = src.index("k_chol_x(DevPlan P")
    body = src[at:src.index("__global__", at)]
    assert "CompSum" in body and "__fmul_rn(" in body
    assert not re.search(r"\w\.x \* \w+\.x", body)      # no product enters a plain float32 sum
    assert "double" not in body.split("CompSum sum[4]")[1]  # and a row needs no float64 sum (two lanes a cycle)
