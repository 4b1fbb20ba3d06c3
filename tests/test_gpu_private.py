"""The row pass with private accumulators against the bundled ring: the same dot
products, so with exact sums (accumulate = 1) the same bits in every mode, on
bundles around every class and register limit, every format, more scenarios than
CTAs' shares and fewer items than CTAs.  With float sums only the order of the
scatter differs."""
import numpy as np
import pytest
import scipy.sparse as sp

from oracle import Weighted
from synthetic import from_dense, random_problem
from tests.gpu_util import gpu_lib, plan_of, fp32_op_bound

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


def _widths_problem(widths, n, N, seed):
    """One bundle (4 rows) per width, whose rows together touch that many spots."""
    rng = np.random.default_rng(seed)
    A = []
    for s in range(N):
        M = np.zeros((4 * len(widths), n), dtype=np.float32)
        for b, w in enumerate(np.roll(widths, s)):
            cols = rng.choice(n, size=w, replace=False)
            for c in cols:
                rows = rng.choice(4, size=int(rng.integers(1, 5)), replace=False)
                M[4 * b + rows, c] = rng.uniform(0.1, 2.0, size=len(rows))
            M[4 * b + np.arange(4), cols[rng.integers(0, w, size=4)]] += 0.5   # no row is empty
        A.append(M)
    m = 4 * len(widths)
    return from_dense(A, rng.uniform(0.1, 5.0, size=m), rng.uniform(0.0, 3.0, size=m), np.zeros(n), np.full(n, 8.0))


CASES = {
    # one more and one fewer than 8 / 16 / 32 lanes take, the slot counts of 32 lanes,
    # their register limit (384) and the doubled tail behind it
    "limits": dict(widths=[1, 2, 7, 8, 9, 15, 16, 17, 47, 48, 49, 64, 65, 95, 96, 97, 128, 129, 160, 161, 192, 224,
                           225, 256, 257, 288, 289, 320, 321, 383, 384, 385, 415, 416, 417, 700], n=701, N=2, seed=1),
    # groups of 16 and 8 lanes that are not full, more scenarios than one share holds
    "many": dict(widths=[50, 50, 50, 10, 10, 10, 10, 10], n=61, N=300, seed=2),
    "one": dict(widths=[3], n=5, N=1, seed=3),
}
FORMS = [(0, 32), (0, 16), (1, 32), (1, 16), (2, 32), (2, 16)]


@pytest.mark.parametrize("case", sorted(CASES))
@pytest.mark.parametrize("fmt,iw", FORMS)
def test_exact_sums_have_the_rings_bits(rpt, case, fmt, iw):
    prob = _widths_problem(**CASES[case])
    rng = np.random.default_rng(5)
    V = rng.normal(size=(prob.N, prob.n))
    x = rng.uniform(0.0, 3.0, size=prob.n)
    got = {}
    for name, kw in (("private", {}), ("ring", dict(ring_threads=1024))):
        with plan_of(rpt, prob, row_path=4, accumulate=1, value_format=fmt, index_width=iw, **kw) as P:
            f, dose = P.objective(x, dose=True)
            z, info = P.admm_bb_solve(max_iter=4, cg_max=6)     # scenarios drop out of the passes one by one
            got[name] = [P.apply_normal(V, 1.3), P.gradient(x)[0], dose, z, np.array([info["inner"]])]
            fs = [f, P.objective(x), P.gradient(x)[1], info["f"]]
        got[name + "_f"] = np.array(fs)
    for a, b in zip(got["private"], got["ring"]):
        assert np.array_equal(a, b)
    # objectives are summed per CTA and so in another order
    np.testing.assert_allclose(got["private_f"], got["ring_f"], rtol=1e-12)


@pytest.mark.parametrize("case", sorted(CASES))
def test_float_sums_match_the_oracle_and_repeat(rpt, case):
    prob = _widths_problem(**CASES[case])
    W = Weighted(prob)
    k = fp32_op_bound(prob)
    V = np.random.default_rng(6).normal(size=(prob.N, prob.n))
    with plan_of(rpt, prob) as P:
        U = [P.apply_normal(V, 0.7) for _ in range(3)]
    assert np.array_equal(U[0], U[1]) and np.array_equal(U[0], U[2])   # fixed shares, fixed turns
    for s in range(0, prob.N, max(1, prob.N // 7)):
        A = abs(W.At[s])
        mag = A.T @ (A @ np.abs(V[s])) + 0.35 * np.abs(V[s])
        assert np.all(np.abs(U[0][s] - W.normal_apply(s, V[s], 0.7)) <= k * mag + 1e-300)


def test_non_finite_vectors_reach_the_result(rpt):
    """Absent block columns of a lane never carry a NaN or an infinity into a sum
    that should be finite, and a vector that is not finite makes the solve report it."""
    prob = random_problem(7, m=400, n=90, N=2, mean_row=20.0)
    with plan_of(rpt, prob) as P:
        V = np.random.default_rng(1).normal(size=(2, 90)) * 1e38     # products overflow to infinity
        U = P.apply_normal(V, 0.0)
        assert not np.all(np.isfinite(U))
        assert np.all(np.isfinite(P.apply_normal(V * 1e-38, 0.0)))   # and leave nothing behind
