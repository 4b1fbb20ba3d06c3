"""Work units of the row pass with private accumulators on the CPU
(paper_2304_14568_gb300/csrc/layout.h, built here with the host compiler): items
cover every bundle once within their lane class, and any run of units holds its
share of the cost to within one item."""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2304_14568_gb300", "csrc")
CUDA_INC = "/usr/local/cuda/include"


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None or not os.path.exists(os.path.join(CUDA_INC, "vector_types.h")):
        pytest.skip("needs g++ and the CUDA headers")
    out = str(tmp_path_factory.mktemp("units") / "libunits_shim.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", "-I", CSRC, "-I", CUDA_INC,
                    os.path.join(HERE, "units_shim.cpp"), "-o", out], check=True)
    L = C.CDLL(out)
    i32p = np.ctypeslib.ndpointer(np.int32, flags="C")
    L.shim_items.argtypes = [i32p, C.c_int, i32p, i32p, i32p]
    L.shim_units.argtypes = [i32p, i32p, C.c_int, C.c_longlong, C.c_int, i32p, C.c_int, i32p, C.POINTER(C.c_int)]
    return L


def _offsets(widths):
    return np.concatenate([[0], np.cumsum(widths)]).astype(np.int32)


def _items(shim, widths):
    cls, q, cnt = np.zeros(3, np.int32), np.zeros(len(widths) + 1, np.int32), np.zeros(len(widths) + 1, np.int32)
    k = shim.shim_items(_offsets(widths), len(widths), cls, q, cnt)
    return cls, q[:k], cnt[:k]


@pytest.mark.parametrize("seed", range(6))
def test_items_cover_every_bundle_in_its_class(shim, seed):
    rng = np.random.default_rng(seed)
    nb = int(rng.integers(0, 60))
    w = np.sort(rng.integers(1, [30, 100, 200, 700, 60, 97][seed], size=nb))[::-1]
    cls, q, cnt = _items(shim, w)
    lanes = np.where(w > 96, 32, np.where(w > 48, 16, 8))      # 6 block columns a lane
    assert cls.tolist() == [int((lanes == g).sum()) for g in (32, 16, 8)]
    assert np.array_equal(np.concatenate([np.arange(a, a + c) for a, c in zip(q, cnt)] + [[]]), np.arange(nb))
    for a, c in zip(q, cnt):
        g = lanes[a]
        assert np.all(lanes[a:a + c] == g) and 1 <= c <= 32 // g


@pytest.mark.parametrize("nb,parts", [((0,), 100), ((1,), 100), ((40, 0, 7), 8), ((300, 200, 100), 640),
                                      ((50, 60), 100000)])
def test_units_share_the_cost(shim, nb, parts):
    rng = np.random.default_rng(sum(nb) + parts)
    widths = [np.sort(np.maximum(1, rng.gamma(1.2, 120.0, size=k)).astype(int))[::-1] for k in nb]
    bpc = 20
    # the cost as layout.h states it
    cost = []
    for w in widths:
        cls, q, cnt = _items(shim, w)
        c = []
        for a, k in zip(q, cnt):
            cols = int(w[a:a + k].sum())
            g = 32 if w[a] > 96 else 16 if w[a] > 48 else 8
            c.append(cols * bpc + (max(0, cols - 384) * 26 if g == 32 else 0) + {32: 3000, 16: 3700, 8: 5300}[g])
        cost.append(np.array(c, dtype=np.int64))
    total = int(sum(c.sum() for c in cost))
    target = max(1, total // parts)
    cap = total // target + len(nb) + 16
    ubeg, uoff, widest = np.zeros(cap, np.int32), np.zeros(len(nb) + 1, np.int32), C.c_int()
    k = shim.shim_units(np.concatenate([_offsets(w) for w in widths]), np.array(nb, np.int32), len(nb), parts, bpc,
                        ubeg, cap, uoff, C.byref(widest))
    assert k >= 0 and uoff[0] == 0 and uoff[-1] == k
    for s, c in enumerate(cost):
        u = ubeg[uoff[s]:uoff[s + 1]]
        if len(c) == 0:
            assert len(u) == 0
            continue
        assert u[0] == 0 and np.all(np.diff(u) >= 0) and u[-1] <= len(c)
        cum = np.concatenate([[0], np.cumsum(c)])
        assert len(u) == -(-int(cum[-1]) // target)
        # a unit begins within one item of its place on the cost axis
        place = target * np.arange(len(u))
        assert np.all(cum[u] >= place) and np.all((u == 0) | (cum[np.maximum(u - 1, 0)] < place))
    if any(nb):
        cols = [int(w[a:a + m].sum()) for w in widths for a, m in zip(*_items(shim, w)[1:])]
        assert widest.value == max(cols)
