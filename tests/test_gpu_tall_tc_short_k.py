"""FP32 regime (i), n > 16, with so few columns of k that a chain of fmas rounds less than the tensor cores' accumulators are
cut: bit for bit the fma kernel's result (tsmm_execute_noalloc), and a single product correctly rounded."""
import numpy as np
import pytest
import torch

import paper_2208_08088_gb300 as tsmm
from gpu_util import to_device

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("k", [1, 2, 7, 15])
@pytest.mark.parametrize("n", [17, 32, 48, 64])
def test_few_columns_are_computed_with_fmas(n, k, pad):
    m = 3001
    rng = np.random.default_rng(23)
    A = np.asfortranarray(rng.uniform(1, 2, (m, k)).astype(np.float32))
    B = np.asfortranarray(rng.uniform(1, 2, (k, n)).astype(np.float32))
    C0 = np.asfortranarray(rng.uniform(-1, 1, (m, n)).astype(np.float32))
    dA, dB = to_device(A, ld=m + pad), to_device(B)
    pb, pl = tsmm.pack_b(dB), tsmm.plan(m, n, k, torch.float32)
    for alpha, beta in ((1.0, 0.0), (0.7, 0.3)):
        C, F = to_device(C0), to_device(C0)
        tsmm.execute(pl, alpha, dA, pb, beta, C)
        pl.check()
        tsmm.tsmm_execute_noalloc(tsmm.F32, m, n, k, alpha, dA.data_ptr(), m + pad, dB.data_ptr(), k, beta, F.data_ptr(), m)
        torch.cuda.synchronize()
        np.testing.assert_array_equal(C.cpu().numpy(), F.cpu().numpy())
        if k == 1 and beta == 0.0:
            np.testing.assert_array_equal(C.cpu().numpy(), A * B)
