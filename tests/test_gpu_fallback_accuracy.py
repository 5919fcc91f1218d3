"""Items that the tensor-core kernels of regime (i) leave to plain fmas: their error (2-norm) is no larger than that of the fma
kernels, which tsmm_execute_noalloc runs, on the same inputs, although an item is one block's and its k range longer."""
import numpy as np
import pytest
import torch

import oracle
import paper_2208_08088_gb300 as tsmm
from gpu_util import to_device

pytestmark = pytest.mark.gpu


def errors(A, B, rows):
    m, k = A.shape
    n = B.shape[1]
    dt, code = (torch.float32, tsmm.F32) if A.dtype == np.float32 else (torch.float64, tsmm.F64)
    dA, dB = to_device(A), to_device(B)
    pb, pl = tsmm.pack_b(dB), tsmm.plan(m, n, k, dt)
    assert pl.info()["bm"] == 128  # a tensor-core plan
    C, F = tsmm.colmajor(m, n, dt), tsmm.colmajor(m, n, dt)
    tsmm.execute(pl, 1.0, dA, pb, 0.0, C)
    pl.check()
    tsmm.tsmm_execute_noalloc(code, m, n, k, 1.0, dA.data_ptr(), m, dB.data_ptr(), k, 0.0, F.data_ptr(), m)
    torch.cuda.synchronize()
    ref, _ = oracle.tsmm(1.0, np.asfortranarray(A[:rows]), B, 0.0, None)
    return [float(np.linalg.norm(X.cpu().numpy()[:rows] - ref) / np.linalg.norm(ref)) for X in (C, F)]


@pytest.mark.parametrize("n", [4, 8, 16, 40, 64])
def test_fp64_steep_columns(n):
    """Columns of A scaled by 10^U[-2,2], rows of B by the inverse: no lower bound of sum|a||b| in sight."""
    k = 2048
    m = -(-40_000_000 // ({40: 48}.get(n, n) * k)) + 1
    rng = np.random.default_rng(19)
    u = rng.uniform(-2, 2, k)
    A = np.asfortranarray(rng.uniform(-1, 1, (m, k)) * 10.0 ** u)
    B = np.asfortranarray(rng.uniform(-1, 1, (k, n)) * 10.0 ** -u[:, None])
    digits, fma = errors(A, B, min(m, 300))
    assert digits <= fma, (digits, fma)


@pytest.mark.parametrize("n", [20, 48, 64])
def test_fp32_infinite_neighbour(n):
    """One infinity in a row of every slab: the slab's other rows are computed with fmas too."""
    m, k = 512, 8192
    rng = np.random.default_rng(20)
    A = rng.uniform(-1, 1, (m, k)).astype(np.float32)
    A[127::128, ::64] = np.inf  # in every item's k range
    A, B = np.asfortranarray(A), np.asfortranarray(rng.uniform(-1, 1, (k, n)).astype(np.float32))
    split, fma = errors(A, B, 127)
    assert split <= fma, (split, fma)
