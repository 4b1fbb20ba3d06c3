"""What the benchmark says about the row pass is what ran: the kernel, its variant
(which keys the stored traffic) and its configuration."""
import numpy as np
import pytest

import bench

RING = dict(row_path=4, exact_sums=0, chunk_entries=4096, chunk_rows=128, stages=3, ring_threads=768)


@pytest.mark.parametrize("st,rp,kernel,variant", [
    (RING, dict(accumulators=4, threads=480, ring_bytes=126464), "k_rowpass_priv", "private-float"),
    (dict(RING, exact_sums=1), dict(accumulators=3, threads=480, ring_bytes=99000), "k_rowpass_priv", "private-exact"),
    (RING, dict(accumulators=0, threads=768, ring_bytes=0), "k_rowpass_tma", "bundled-float-768t"),
    (dict(RING, exact_sums=1, ring_threads=1024), dict(accumulators=0, threads=1024, ring_bytes=0), "k_rowpass_tma",
     "bundled-exact"),
    (dict(RING, row_path=2), dict(accumulators=0, threads=1024, ring_bytes=0), "k_rowpass_tma", "ring"),
])
def test_report(st, rp, kernel, variant):
    k, v, cfg = bench.row_pass_report(st, rp)
    assert (k, v) == (kernel, variant)
    assert cfg["threads"] == rp["threads"]
    assert ("private_accumulators" in cfg) == (rp["accumulators"] > 0) == ("chunk_entries" not in cfg)


@pytest.mark.gpu
@pytest.mark.parametrize("n,exact,accs", [(60, 0, 6), (60, 1, 6), (5000, 0, 4), (5000, 1, 0), (7000, 0, 3),
                                          (9500, 0, 2), (12000, 0, 0)])
def test_query_on_plans(n, exact, accs):
    """Accumulators by width: the most of 6, 4, 3, 2 that leave a ring of 96 KB (three at
    least for exact sums), none on plans that set the ring's threads."""
    from synthetic import random_problem
    from tests.gpu_util import gpu_lib, plan_of
    rpt = gpu_lib()
    prob = random_problem(3, m=200, n=n, N=1, mean_row=6.0, long_rows=0)   # (a row as wide as the plan fits no stage)
    with plan_of(rpt, prob, row_path=4, accumulate=1 if exact else 2) as P:
        rp = P.row_pass()
        assert rp["accumulators"] == accs
        assert rp["threads"] == (480 if accs else P.stats()["ring_threads"])
        assert (rp["ring_bytes"] >= 98304) == (accs > 0)
        assert np.all(np.isfinite(P.apply_normal(np.ones((1, n)))))
    with plan_of(rpt, random_problem(3, m=200, n=60, N=1, mean_row=6.0), row_path=4, ring_threads=768) as P:
        assert P.row_pass() == dict(accumulators=0, threads=768, ring_bytes=0)
