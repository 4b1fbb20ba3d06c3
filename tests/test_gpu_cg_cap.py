"""CG loops that end at their cap: the loop's body holds two steps, and a step past
the cap must neither change an iterate nor run a row pass over active scenarios."""
import numpy as np
import pytest

from synthetic import random_problem
from tests.gpu_util import gpu_lib, plan_of

pytestmark = pytest.mark.gpu
TIGHT = dict(eps_abs=0.0, eps_rel=0.0, cg_theta=1e-12, cg_eta0=1e-12, cg_floor_rel=0.0)


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


@pytest.mark.parametrize("n", [40, 300])
@pytest.mark.parametrize("cg_max", [1, 2, 3, 4, 9, 11])
def test_graph_and_host_loop_agree_at_the_cap(rpt, n, cg_max):
    """With exact sums the graph's loop and the host's loop, which makes one step at a
    time, give the same bits and the same counts."""
    prob = random_problem(41, m=500, n=n, N=3, mean_row=12.0, ub=6.0)
    with plan_of(rpt, prob, accumulate=1) as P:
        got = []
        for graph in (1, 0):
            _, info = P.admm_bb_solve(max_iter=5, cg_max=cg_max, use_graph=graph, **TIGHT)
            got.append((P.state_get(), info["inner"], info["row_passes"], info["kernels"]))
    for a, b in zip(got[0][0], got[1][0]):
        assert np.array_equal(a, b)
    assert got[0][1:] == got[1][1:]
    assert got[0][1] == 5 * cg_max * prob.N                # no loop ended before its cap


def test_no_row_pass_is_thrown_away_at_a_cap_of_one(rpt):
    """An iteration at cap 1 makes two passes (residual, one step), at cap 2 three; on a
    plan whose passes take most of the time it is at most 2/3 plus the vector kernels'
    share.  A pass thrown away at cap 1 would make the two alike."""
    rng = np.random.default_rng(3)
    m, n, N, width = 120_000, 1000, 4, 64
    row_ptr = (np.arange(m + 1, dtype=np.int64) * width).astype(np.int32)
    problem = dict(m=m, n=n, N=N, row_ptr=[], col_idx=[], val=[])
    for _ in range(N):
        start = rng.integers(0, n - width, size=m)
        problem["row_ptr"].append(row_ptr)
        problem["col_idx"].append((start[:, None] + np.arange(width)).astype(np.int32).ravel())
        problem["val"].append(rng.uniform(0.1, 1.0, size=m * width).astype(np.float32))
    args = [problem[k] for k in ("m", "n", "N", "row_ptr", "col_idx", "val")]
    with rpt.Plan(*args, rng.uniform(0.5, 2.0, size=m), rng.uniform(0.0, 3.0, size=m), lb=np.zeros(n),
                  ub=np.full(n, 8.0)) as P:
        def best(cg_max):
            return min(P.admm_bb_solve(max_iter=30, cg_max=cg_max, **TIGHT)[1]["seconds"] for _ in range(6))
        best(1), best(2)
        t1, t2 = best(1), best(2)
    print(f"30 iterations: cap 1 {1e3 * t1:.2f} ms, cap 2 {1e3 * t2:.2f} ms, ratio {t1 / t2:.2f}")
    assert t1 < 0.82 * t2, (t1, t2)
