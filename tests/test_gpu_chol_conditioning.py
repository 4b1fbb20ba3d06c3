"""The cached factor on ill-conditioned B_s (nearly dependent spots, small penalty):
rows below a diagonal block and the inverse are products with inverted diagonal
blocks on the tensor cores (three-term TF32), so their error is held against a plain
FP32 factorisation, inverse and product of the same B_s (LAPACK's spotrf, spotri)."""
import numpy as np
import pytest
from scipy.linalg import lapack

from tests.gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


def _near_dependent(n, eps, seed):
    """m x n: pairs of columns that differ by eps, relatively."""
    rng = np.random.default_rng(seed)
    m = 3 * n
    A = rng.uniform(0.1, 1.0, size=(m, n)) * (rng.random((m, n)) < 0.3)
    h = n // 2
    A[:, 1::2] = A[:, 0:2 * h:2] * (1.0 + eps * rng.normal(size=(m, h)))
    return np.abs(A).astype(np.float32), rng.uniform(0.5, 2.0, size=m), rng.uniform(0.0, 3.0, size=m)


@pytest.mark.parametrize("n", [48, 64, 130, 301])
@pytest.mark.parametrize("eps,rho_scale,least", [(1e-1, 1e-2, 5e2), (1e-2, 1e-3, 5e3), (3e-3, 1e-4, 5e4)])
def test_error_of_a_plain_fp32_factor(rpt, n, eps, rho_scale, least):
    """Mean error over five matrices within four times the plain one's: both are a few
    rounding errors times the condition number; here B_s is summed by atomics, one row
    block after another, and the inverse's three products each drop a term of 2^-22."""
    err, ref = [], []
    for seed in range(5):
        A, w, p = _near_dependent(n, eps, seed)
        m = A.shape[0]
        A64 = A.astype(np.float64)
        G = A64.T @ (w[:, None] * A64)
        rho = rho_scale * 2.0 * np.trace(G) / n
        B = G + 0.5 * rho * np.eye(n)
        c = A64.T @ (w * p)
        x = np.linalg.solve(B, c)
        assert np.linalg.cond(B) > least
        S = (np.sqrt(w)[:, None] * A64).astype(np.float32)
        L, info = lapack.spotrf(S.T @ S + np.float32(0.5 * rho) * np.eye(n, dtype=np.float32), lower=1)
        assert info == 0
        inv, info = lapack.spotri(L, lower=1)
        inv = np.tril(inv) + np.tril(inv, -1).T
        ref.append(np.linalg.norm(inv.astype(np.float64) @ c.astype(np.float32).astype(np.float64) - x) /
                   np.linalg.norm(x))
        rows = [np.flatnonzero(A[i]).astype(np.int32) for i in range(m)]
        rp = np.concatenate([[0], np.cumsum([r.size for r in rows])]).astype(np.int32)
        with rpt.Plan(m, n, 1, [rp], [np.concatenate(rows)], [np.concatenate([A[i, r] for i, r in enumerate(rows)])],
                      w, p) as P:
            P.admm_bb_solve(rho=rho, max_iter=1, eps_abs=0.0, eps_rel=0.0, subproblem=rpt.SUB_CHOL)
            X = np.asarray(P.state_get()[1]).reshape(-1)
        err.append(np.linalg.norm(X - x) / np.linalg.norm(x))
    print(f"n {n} eps {eps}: error {np.mean(err):.2e}, plain FP32 {np.mean(ref):.2e}")
    assert np.mean(err) <= 4.0 * np.mean(ref)
