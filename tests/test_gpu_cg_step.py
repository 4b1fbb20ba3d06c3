"""The CG step at every width of its thread-block cluster (1, 2, 4, 8 CTAs, more
than one row of threads a CTA): iterates against the oracle's exact subproblems
with the error budget of test_gpu_admm, and, with exact sums, the same bits on
every run: the CTAs' parts of the step's inner products all arrive."""
import math

import numpy as np
import pytest

from oracle import Weighted, admm_bb, default_rho
from synthetic import random_problem
from tests.gpu_util import fp32_op_bound, gpu_lib, plan_of

pytestmark = pytest.mark.gpu
TIGHT_CG = dict(cg_theta=1e-12, cg_eta0=1e-12, cg_floor_rel=0.0, cg_max=200)


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


@pytest.mark.parametrize("n", [256, 257, 513, 1025, 2049])
def test_iterates_at_every_cluster_width(rpt, n):
    prob = random_problem(37, m=500, n=n, N=3, mean_row=30.0, long_rows=0, ub=6.0)
    W = Weighted(prob)
    rho = 0.3 * default_rho(W)
    k = 2
    ref = admm_bb(W, rho=rho, max_iter=k, eps_abs=0.0, eps_rel=0.0)
    e2 = 0.0
    for s in range(prob.N):
        xs = np.abs(ref["x"][s])
        Aa = abs(W.At[s])
        e2 += float(np.sum((Aa.T @ (Aa @ xs) + 0.5 * rho * xs + np.abs(W.b(s))) ** 2))
    bound = 10.0 * k * (2.0 / rho) * fp32_op_bound(prob) * math.sqrt(e2)
    runs = []
    with plan_of(rpt, prob, accumulate=1) as P:
        for _ in range(4):
            P.admm_bb_solve(rho=rho, max_iter=k, eps_abs=0.0, eps_rel=0.0, **TIGHT_CG)
            runs.append(P.state_get())
    z, X, Y = runs[0]
    assert np.linalg.norm(X - ref["x"]) <= bound
    assert np.linalg.norm(z - ref["z"]) <= bound
    assert np.linalg.norm(Y - ref["y"]) <= 4.0 * rho * bound + 1e-9 * np.linalg.norm(ref["y"])
    for again in runs[1:]:
        for a, b in zip(again, runs[0]):
            assert np.array_equal(a, b)
