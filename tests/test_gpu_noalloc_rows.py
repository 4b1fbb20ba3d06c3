"""The allocation-free operator on matrices of few and of long rows, around the number of
rows that each get a warp (8192) and the entries that a warp and eight lanes keep in
registers (512, 128): against a float64 product within the float32 bound, and the time of
a few long rows beside that of one."""
import numpy as np
import pytest
import scipy.sparse as sp

from tests.gpu_util import EPS32, gpu_lib

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rpt():
    return gpu_lib()


def _rows(lens, n, seed):
    """Rows of the given lengths, each on one window of the spots."""
    rng = np.random.default_rng(seed)
    lens = np.asarray(lens)
    rp = np.concatenate([[0], np.cumsum(lens)]).astype(np.int32)
    start = np.repeat(rng.integers(0, n - lens + 1), lens)
    ci = (np.arange(rp[-1]) - np.repeat(rp[:-1], lens) + start).astype(np.int32)
    return rp, ci, rng.uniform(0.1, 1.0, size=int(rp[-1])).astype(np.float32)


def _on_device(rpt, n, rp, ci, va, w, V):
    import torch
    d = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (rp, ci, va, w, V)]
    u = torch.empty(n, dtype=torch.float32, device="cuda")
    stream = torch.cuda.current_stream().cuda_stream

    def call():
        rpt.normal_apply_noalloc(len(rp) - 1, n, *[t.data_ptr() for t in d], 1.4, u.data_ptr(), stream)
        return u
    return call


@pytest.mark.parametrize("lens,n", [
    ([1], 1), ([0, 0, 5], 40), ([127, 128, 129, 511, 512, 513, 767, 768, 769, 4000], 4000),
    ([8000] * 3 + [0] * 50 + [1] * 7, 8192), (np.arange(700) % 300, 500), (np.arange(8191) % 160, 300),
    (np.arange(8192) % 160, 300), (np.arange(8193) % 160, 300), (np.arange(9000) % 3 * 260, 1000),
])
def test_rows_of_every_kind(rpt, lens, n):
    rp, ci, va = _rows(lens, n, 3)
    m = len(rp) - 1
    rng = np.random.default_rng(4)
    w, V = rng.uniform(0.1, 2.0, size=m).astype(np.float32), rng.normal(size=n).astype(np.float32)
    got = _on_device(rpt, n, rp, ci, va, w, V)().cpu().numpy().astype(np.float64)
    A = sp.csr_matrix((va.astype(np.float64), ci, rp), shape=(m, n))
    ref = A.T @ (w.astype(np.float64) * (A @ V)) + 0.7 * V
    mag = A.T @ (w * (A @ np.abs(V))) + 0.7 * np.abs(V)
    K = int(np.bincount(ci, minlength=n).max(initial=0)) + int(np.diff(rp).max(initial=0)) + 8
    assert np.all(np.abs(got - ref) <= K * EPS32 * mag)


def test_a_few_long_rows_take_little_longer_than_one(rpt):
    """Each row has a warp of its own: 100 rows of 8000 entries wait for one row's chain,
    not for several one after another (a few times as long)."""
    import torch
    n = 8000
    t = []
    for m in (1, 100):
        rp, ci, va = _rows([8000] * m, n, 5)
        call = _on_device(rpt, n, rp, ci, va, np.ones(m, np.float32), np.ones(n, np.float32))
        best = 1e9
        for _ in range(8):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            for _ in range(10):
                call()
            e1.record()
            torch.cuda.synchronize()
            best = min(best, e0.elapsed_time(e1) / 10)
        t.append(1e3 * best)
    print(f"one row {t[0]:.1f} us, 100 rows {t[1]:.1f} us")
    assert t[1] < 2.5 * t[0]
