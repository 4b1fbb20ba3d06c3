"""The choice between private accumulators and the ring (csrc/layout.h) on the CPU, at
shapes where both sides were measured: the pass that was faster is the one taken."""
import ctypes as C
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2304_14568_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"
F32, BF16, FP8 = 0, 1, 2


@pytest.fixture(scope="module")
def pays(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "vector_types.h")):
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("passrule") / "libpassrule_shim.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I", CSRC, "-I", CUDA_INC,
                    os.path.join(HERE, "passrule_shim.cpp"), "-o", out], check=True)
    f = C.CDLL(out).shim_private_sums_pay
    f.argtypes = [C.c_int, C.c_int, C.c_int, C.c_longlong, C.c_longlong, C.c_int]
    return f


# accumulators, exact, format, block columns (millions, over 152 CTAs), columns a bundle, the
# ring's stage, microseconds of the pass with private accumulators and of the ring
MEASURED = [
    (2, 0, BF16, 42.04, 195, 4096, 219.2, 169.6), (2, 0, FP8, 42.04, 195, 4096, 207.7, 179.1),
    (2, 0, F32, 42.04, 195, 3072, 245.1, 209.5), (2, 0, BF16, 9.78, 197, 4096, 59.7, 54.5),
    (2, 0, F32, 9.78, 197, 3072, 67.6, 63.7), (2, 0, BF16, 40.96, 308, 4096, 207.9, 182.4),
    (2, 0, BF16, 17.77, 312, 4096, 98.0, 91.1), (2, 0, F32, 17.77, 312, 3072, 110.5, 113.9),
    (2, 0, FP8, 17.77, 312, 4096, 94.9, 95.9), (2, 0, BF16, 5.97, 311, 4096, 38.4, 41.6),
    (2, 0, F32, 1.83, 123, 3072, 20.5, 26.6), (2, 0, BF16, 13.64, 428, 4096, 82.7, 89.9),
    (2, 0, F32, 26.24, 414, 3072, 164.4, 186.1), (2, 0, F32, 47.33, 356, 2048, 256.3, 429.4),
    (3, 0, BF16, 28.24, 136, 4096, 115.8, 118.1), (3, 0, F32, 37.37, 174, 3072, 159.8, 185.4),
    (4, 0, F32, 28.03, 130, 3072, 121.4, 127.9), (6, 0, F32, 0.72, 50, 4096, 10.3, 26.8),
    (3, 1, FP8, 17.68, 86, 4096, 123.4, 110.9), (4, 1, FP8, 25.36, 102, 4096, 159.4, 151.8),
    (3, 1, FP8, 4.50, 88, 4096, 40.3, 38.5), (4, 1, FP8, 2.67, 86, 4096, 26.7, 38.9),
    (6, 1, FP8, 16.61, 148, 4096, 98.2, 113.0), (3, 1, F32, 17.68, 86, 3072, 113.8, 124.5),
    (4, 1, BF16, 25.36, 102, 4096, 133.9, 145.5),
]


@pytest.mark.parametrize("accs,exact,fmt,mcols,width,ring_cols,private,ring", MEASURED)
def test_the_faster_pass_is_taken(pays, accs, exact, fmt, mcols, width, ring_cols, private, ring):
    assert bool(pays(accs, exact, fmt, int(mcols * 1e6 / 152), width, ring_cols)) == (private < ring)


def test_edges(pays):
    assert pays(2, 0, F32, 40000, 10, 4096) and not pays(2, 0, F32, 40001, 299, 3072)
    assert pays(2, 0, F32, 40001, 300, 3072) and pays(2, 0, F32, 40001, 10, 3071)
    assert not pays(2, 0, BF16, 40001, 399, 3072) and pays(2, 0, BF16, 40001, 400, 3072)
    assert pays(3, 1, FP8, 20000, 10, 4096) and not pays(4, 1, FP8, 20001, 700, 512)
    assert pays(3, 1, BF16, 10 ** 9, 10, 4096) and pays(6, 1, FP8, 10 ** 9, 10, 4096)
