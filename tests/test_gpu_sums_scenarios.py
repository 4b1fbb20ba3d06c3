"""Sums over row-pass partials and over scenarios at the edges of their batches: scenario
counts around the thread rows that share them and the eight that the consensus step
loads together, wide plans of one scenario, with exact sums bit for bit repeatable and
against float64; and the time of a wide plan's gradient beside its operator's."""
import numpy as np
import pytest

from oracle import Weighted, admm_bb, default_rho
from synthetic import random_problem
from tests.gpu_util import fp32_op_bound, gpu_lib, plan_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


@pytest.mark.parametrize("path,acc", [(4, 2), (4, 1), (2, 0)])
@pytest.mark.parametrize("N,n", [(1, 33), (2, 600), (7, 97), (8, 64), (9, 64), (15, 40), (16, 40), (17, 40), (33, 31)])
def test_gradient_and_consensus_over_scenarios(rpt, N, n, path, acc):
    prob = random_problem(47, m=160, n=n, N=N, mean_row=8.0, ub=6.0)
    W = Weighted(prob)
    x = np.random.default_rng(1).uniform(0.0, 3.0, size=n)
    k = fp32_op_bound(prob)
    g_ref, g_mag = np.zeros(n), np.zeros(n)
    for s in range(N):
        A, b = W.At[s], W.b(s)
        g_ref += 2.0 * (A.T @ (A @ x) - b)
        Aa = abs(A)
        g_mag += 2.0 * (Aa.T @ (Aa @ np.abs(x)) + np.abs(b))
    rho = default_rho(W)
    ref = admm_bb(W, rho=rho, max_iter=2, eps_abs=0.0, eps_rel=0.0, subproblem="chol")
    with plan_of(rpt, prob, row_path=path, accumulate=acc) as P:
        g = [np.asarray(P.gradient(x)[0]) for _ in range(2)]
        P.admm_bb_solve(rho=rho, max_iter=2, eps_abs=0.0, eps_rel=0.0, subproblem=rpt.SUB_CHOL)
        z, X, _ = P.state_get()
    assert np.all(np.abs(g[0] - g_ref) <= k * g_mag + 1e-300)
    if acc == 1:
        assert np.array_equal(g[0], g[1])
    np.testing.assert_allclose(z, ref["z"], rtol=1e-4, atol=1e-5 * np.abs(ref["z"]).max())


def test_a_wide_plans_gradient_takes_little_longer_than_its_operator(rpt):
    """20,000 spots, one scenario (the ring with its slot lists): the gradient is the
    operator's pass and a sum over the same partials; loads that wait for one another, or
    blocks of mostly idle warps in a second wave, made it twice as long."""
    import time
    prob = random_problem(49, m=20_000, n=20_000, N=1, mean_row=40.0, long_rows=0)
    x = np.random.default_rng(1).uniform(0.0, 3.0, size=prob.n)

    def best(f):
        f()
        t = []
        for _ in range(30):
            t0 = time.perf_counter()
            f()
            t.append(time.perf_counter() - t0)
        return 1e6 * min(t)

    with plan_of(rpt, prob, row_path=4) as P:
        a, b = best(lambda: P.apply_normal(x, 1.0)), best(lambda: P.gradient(x))
    print(f"operator {a:.0f} us, gradient {b:.0f} us")
    assert b < 1.35 * a
