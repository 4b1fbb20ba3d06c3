"""Doses of large volumes with few voxels in the beams: the caller's array is filled
in pieces through a bounded buffer, so the plan does not hold 8 N m bytes."""
import numpy as np
import pytest
import scipy.sparse as sp

from tests.gpu_util import gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


def _sparse_volume(m, n, N, rows, seed):
    """N matrices of m rows of which `rows` (the first and the last among them) have entries."""
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(N):
        at = np.unique(np.concatenate([[0, m - 1], rng.integers(0, m, size=rows)]))
        A = sp.csr_matrix((rng.uniform(0.1, 1.0, size=5 * at.size).astype(np.float32),
                           (np.repeat(at, 5), np.concatenate([rng.choice(n, 5, replace=False) for _ in at]))),
                          shape=(m, n))
        A.sort_indices()
        out.append(A)
    return out


# pieces of several scenarios, of parts of one, and one piece for all
@pytest.mark.parametrize("m,N", [(1_500_000, 13), (5_000_000, 2), (2_000, 3)])
def test_doses_in_pieces_and_bounded_memory(rpt, m, N):
    import torch
    n = 40
    A = _sparse_volume(m, n, N, 300, 11)
    x = np.random.default_rng(2).uniform(0.0, 3.0, size=n)
    w, p = np.ones(m), np.zeros(m)
    with rpt.Plan(m, n, N, [a.indptr.astype(np.int32) for a in A], [a.indices.astype(np.int32) for a in A],
                  [a.data for a in A], w, p) as P:
        P.objective(x)
        free0 = torch.cuda.mem_get_info()[0]
        got = [P.objective(x, dose=True) for _ in range(2)]
        held = free0 - torch.cuda.mem_get_info()[0]
    kept = np.unique(np.concatenate([np.flatnonzero(np.diff(a.indptr)) for a in A])).size
    # the pass's doses, an index of the voxels, the buffer of 32 MB, and two allocation granules
    assert held <= 4 * N * kept + 4 * m + (32 << 20) + (4 << 20), held
    for f, dose in got:
        dose = np.asarray(dose).reshape(N, m)
        for s in range(N):
            ref = A[s].astype(np.float64) @ x
            assert np.array_equal(dose[s] != 0, ref != 0)
            np.testing.assert_allclose(dose[s], ref, rtol=1e-5)
        assert f == pytest.approx(sum(float(((a.astype(np.float64) @ x) ** 2).sum()) for a in A), rel=1e-5)
    assert np.array_equal(np.asarray(got[0][1]), np.asarray(got[1][1]))
