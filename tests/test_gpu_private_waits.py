"""The waits of the row pass with private accumulators when they run out: the call
reports it, nothing hangs and the context stays usable (no GPU fault is made: the
testing hook withholds the turns on the accumulators)."""
import numpy as np
import pytest

from tests.gpu_util import gpu_lib, plan_of
from tests.test_gpu_private import CASES, _widths_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


@pytest.mark.parametrize("acc", [1, 2])
def test_a_turn_that_never_comes_is_reported(rpt, acc):
    prob = _widths_problem(**CASES["limits"])
    V = np.random.default_rng(8).normal(size=(prob.N, prob.n))
    with plan_of(rpt, prob, row_path=4, accumulate=acc, inject_timeout=2) as P:
        with pytest.raises(rpt.RptError) as e:
            P.apply_normal(V, 0.0)
        assert e.value.status == rpt.TIMEOUT and "code 4" in str(e.value)
        assert np.isfinite(P.objective(np.ones(prob.n)))      # a pass without accumulators
    with plan_of(rpt, prob, row_path=4, accumulate=acc) as P:
        assert np.all(np.isfinite(P.apply_normal(V, 0.0)))
