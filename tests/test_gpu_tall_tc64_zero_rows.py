"""FP64 regime (i) on the tensor cores with rows of A that are zero, or whose first nonzero entry comes late: exact values,
and no more than twice the time of a dense A."""
import numpy as np
import pytest
import torch

import paper_2208_08088_gb300 as tsmm
from gpu_util import run, to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("late", [0.0, -0.0, 3.0, 2.0 ** -450, 2.0 ** -1042, 5e-324])
@pytest.mark.parametrize("n,m,k", [(4, 320, 32768), (20, 130, 33000), (64, 256, 32768)])
def test_zero_rows_and_late_entries(n, m, k, late, pad):
    rng = np.random.default_rng(37)
    A = np.asfortranarray(rng.integers(-8, 9, (m, k)).astype(np.float64))
    B = np.asfortranarray(rng.integers(-8, 9, (k, n)).astype(np.float64))
    A[7::128] = 0.0
    A[100:110] = 0.0
    A[107, k - 1 - np.arange(3)] = late  # in two steps of 16 columns at most, the last
    C, pl, _ = run(A, B, None, 1.0, 0.0, lda=m + pad)
    assert pl.info()["bm"] == 128
    np.testing.assert_array_equal(C, A @ B)


def test_zero_rows_take_no_longer():
    m, n, k = 8192, 4, 16384
    A = tsmm.colmajor(m, k, torch.float64)
    A.uniform_(-1, 1)
    B = to_device(np.asfortranarray(np.random.default_rng(1).uniform(-1, 1, (k, n))))
    C = tsmm.colmajor(m, n, torch.float64)
    pb, pl = tsmm.pack_b(B), tsmm.plan(m, n, k, torch.float64)

    def best():
        times = []
        for _ in range(6):
            a, b = torch.cuda.Event(True), torch.cuda.Event(True)
            a.record()
            tsmm.execute(pl, 1.0, A, pb, 0.0, C)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        pl.check()
        return min(times)

    dense = best()
    A[7::128] = 0.0
    assert best() < 2 * dense
