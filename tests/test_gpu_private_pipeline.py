"""The row pass with private accumulators on shares that recycle its pipeline: several
hundred items a CTA, so that the ring of bytes wraps and skips its end many times, the
128 descriptors and their barriers are used again (parity and generation above one) and
the bound on items in flight is met; bundles of every class and beyond the registers'
limit; every number of accumulators.  Exact sums must have the ring kernel's bits;
float sums stay within the float32 bound of a float64 product and repeat bit for bit."""
import numpy as np
import pytest
import scipy.sparse as sp

from tests.gpu_util import EPS32, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


def _matrix(widths, n, seed):
    """Four rows per width on one window of that many spots, a fifth of the entries
    missing (never a row's first, so no row is empty)."""
    rng = np.random.default_rng(seed)
    w4 = np.repeat(widths, 4)
    start = np.repeat(rng.integers(0, n - widths + 1), 4)
    ptr = np.concatenate([[0], np.cumsum(w4)])
    col = np.arange(ptr[-1]) - np.repeat(ptr[:-1] - start, w4)
    keep = rng.random(ptr[-1]) < 0.8
    keep[ptr[:-1]] = True
    rp = np.concatenate([[0], np.cumsum(np.add.reduceat(keep, ptr[:-1]))])
    val = rng.uniform(0.1, 2.0, size=int(rp[-1])).astype(np.float32)
    return rp.astype(np.int32), col[keep].astype(np.int32), val


def _short(n, seed):
    """250,000 bundles of 8 and 16 lanes: about 450 items a CTA of 152."""
    return _matrix(np.random.default_rng(seed).integers(6, 97, size=250_000), n, seed)


def _wide(n, seed):
    """15,000 bundles of 32 lanes, a quarter of them past 384 columns: 100 items a CTA, 0.8 MB
    through a ring of 100 to 130 KB (half as much in BF16)."""
    rng = np.random.default_rng(seed)
    return _matrix(np.concatenate([rng.integers(97, 385, size=11_000), rng.integers(385, 800, size=4_000)]), n, seed)


def _wide_fp8(n, seed):
    """As many as exact FP8 sums take with fewer than six accumulators (20,000 columns a CTA)."""
    rng = np.random.default_rng(seed)
    return _matrix(np.concatenate([rng.integers(97, 385, size=6_000), rng.integers(385, 800, size=2_200)]), n, seed)


def _plan(rpt, mats, n, **kw):
    m = len(mats[0][0]) - 1
    rng = np.random.default_rng(9)
    w, p = rng.uniform(0.1, 5.0, size=m), rng.uniform(0.0, 3.0, size=m)
    return rpt.Plan(m, n, len(mats), [a[0] for a in mats], [a[1] for a in mats], [a[2] for a in mats], w, p,
                    lb=np.zeros(n), ub=np.full(n, 8.0), row_path=4, **kw), w


@pytest.fixture(scope="module")
def matrices():
    # spots, accumulators of exact sums, matrices (two scenarios of the short bundles)
    return {"short": (250, 6, [_short(250, 1), _short(250, 2)]), "wide4": (3400, 4, [_wide(3400, 3)]),
            "wide3": (4500, 3, [_wide(4500, 4)]), "wide4_fp8": (3400, 4, [_wide_fp8(3400, 3)]),
            "wide3_fp8": (4500, 3, [_wide_fp8(4500, 4)])}


@pytest.mark.parametrize("case", ["short", "wide4", "wide3"])
@pytest.mark.parametrize("fmt,iw", [(0, 32), (0, 16), (1, 32), (1, 16), (2, 32), (2, 16)])
def test_exact_sums_have_the_rings_bits(rpt, matrices, case, fmt, iw):
    n, accs, mats = matrices[case + ("_fp8" if fmt == 2 and case != "short" else "")]
    N = len(mats)
    rng = np.random.default_rng(5)
    V = rng.normal(size=(N, n))
    x = rng.uniform(0.0, 3.0, size=n)
    got, fs = [], []
    for kw in ({}, dict(ring_threads=1024)):
        P, _ = _plan(rpt, mats, n, accumulate=1, value_format=fmt, index_width=iw, **kw)
        with P:
            assert P.row_pass()["accumulators"] == (0 if kw else accs)
            f, dose = P.objective(x, dose=True)
            g, fg = P.gradient(x)
            got.append([P.apply_normal(V, 1.3), g, dose, P.apply_normal(V, 1.3)])
            fs.append([f, fg])
    for a, b in zip(*got):
        assert np.array_equal(a, b)
    assert np.array_equal(got[0][0], got[0][3])
    np.testing.assert_allclose(fs[0], fs[1], rtol=1e-12)


@pytest.mark.parametrize("fmt,exact,n,accs", [(0, 0, 9000, 0), (1, 0, 9000, 0), (2, 0, 9000, 0), (2, 1, 3400, 0),
                                              (0, 1, 3400, 4), (1, 0, 7000, 3)])
def test_narrow_bundles_keep_the_ring_where_it_is_faster(rpt, fmt, exact, n, accs):
    """8 M block columns of 100 a bundle on average: two accumulators, and FP8's exact sums
    with fewer than six, would wait for turns longer than the ring's atomics take."""
    rp, ci, va = _matrix(np.random.default_rng(1).integers(60, 141, size=82_000), n, 8)
    P, w = _plan(rpt, [(rp, ci, va)], n, accumulate=1 if exact else 2, value_format=fmt, index_width=16)
    with P:
        assert P.stats()["block_cols"] / 152 > 40_000
        assert P.row_pass()["accumulators"] == accs
        V = np.random.default_rng(6).normal(size=n)
        U = np.asarray(P.apply_normal(V, 0.7)).reshape(-1)
    if fmt == 0:
        A = sp.csr_matrix((va.astype(np.float64), ci, rp), shape=(len(rp) - 1, n))
        ref = A.T @ (w * (A @ V)) + 0.35 * V
        assert np.linalg.norm(U - ref) <= 1e-5 * np.linalg.norm(ref)


@pytest.mark.parametrize("n,accs,make", [(250, 6, _short), (4500, 6, _wide), (5000, 4, _wide), (7000, 3, _wide),
                                         (9500, 2, _wide)])
def test_float_sums_by_accumulators(rpt, n, accs, make):
    rp, ci, va = make(n, 6)
    m = len(rp) - 1
    V = np.random.default_rng(6).normal(size=n)
    P, w = _plan(rpt, [(rp, ci, va)], n, accumulate=2)
    with P:
        assert P.row_pass()["accumulators"] == accs
        U = [np.asarray(P.apply_normal(V, 0.7)).reshape(-1) for _ in range(3)]
    assert np.array_equal(U[0], U[1]) and np.array_equal(U[0], U[2])   # fixed shares, fixed turns
    A = sp.csr_matrix((va.astype(np.float64), ci, rp), shape=(m, n))
    ref = A.T @ (w * (A @ V)) + 0.35 * V
    mag = A.T @ (w * (A @ np.abs(V))) + 0.35 * np.abs(V)
    bound = (int(np.diff(rp).max()) + int(np.bincount(ci, minlength=n).max()) + 8) * EPS32
    assert np.all(np.abs(U[0] - ref) <= bound * mag)
    # and much closer than the bound in practice: the errors of a few thousand additions, not of their worst case
    assert np.linalg.norm(U[0] - ref) <= 1e-5 * np.linalg.norm(ref)
