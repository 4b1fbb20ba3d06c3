"""Device memory that a plan keeps after a cached-factor solve: the factor, and a
workspace of at most 128 MB; a larger one is given back."""
import numpy as np
import pytest

from synthetic import random_problem
from tests.gpu_util import gpu_lib, plan_of

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


@pytest.mark.parametrize("n,N,kept", [(600, 3, True), (2050, 9, False)])
def test_memory_held_after_the_factor_is_formed(rpt, n, N, kept):
    import torch
    prob = random_problem(43, m=300, n=n, N=N, mean_row=20.0, ub=6.0)
    with plan_of(rpt, prob) as P:
        P.admm_bb_solve(max_iter=1)                    # everything else a solve allocates
        free0 = torch.cuda.mem_get_info()[0]
        for scale in (1.0, 2.0, 1.0):                  # the factor formed three times
            z, info = P.admm_bb_solve(max_iter=3, subproblem=rpt.SUB_CHOL, rho_scale=scale)
            assert info["setup_seconds"] > 0 and np.all(np.isfinite(z))
            held = free0 - torch.cuda.mem_get_info()[0]
            factor = 4 * N * n * ((n + 3) // 4 * 4)
            assert factor <= held + (2 << 20)
            assert held <= (2 if kept else 1) * factor + 8 * N * n + (8 << 20), (held, factor)
