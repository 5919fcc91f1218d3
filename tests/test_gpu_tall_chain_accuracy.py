"""FP32 regime (i) up to 16 columns: the planner's few splits do not lengthen the chains of fmas.  The error (2-norm) is no
larger than that of chains of 32 columns on 32 splits, two warps to each, restated here."""
import numpy as np
import pytest

from gpu_util import run

pytestmark = pytest.mark.gpu


def chains_of_32(A, B):
    k = A.shape[1]
    part = np.zeros((k // 32, A.shape[0], B.shape[1]), np.float32)
    for p in range(32):  # fma: the exact product, one rounding (in 64 bits first, which changes nothing that shows)
        a, b = A[:, p::32].astype(np.float64), B[p::32].astype(np.float64)
        part = (a.T[:, :, None] * b[:, None, :] + part).astype(np.float32)
    out = np.zeros(part.shape[1:], np.float32)
    for s in range(0, k // 32, 2):
        out = out + (part[s] + part[s + 1])
    return out


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("n", [1, 4, 8, 16])
def test_error_is_that_of_short_chains(n, pad):
    m = k = 2048
    rng = np.random.default_rng(43)
    A = np.asfortranarray(rng.uniform(-1, 1, (m, k)).astype(np.float32))
    B = np.asfortranarray(rng.uniform(-1, 1, (k, n)).astype(np.float32))
    C, _, _ = run(A, B, None, 1.0, 0.0, lda=m + pad)
    ref = A.astype(np.float64) @ B.astype(np.float64)
    want = np.linalg.norm(chains_of_32(A[:512], B) - ref[:512]) / np.linalg.norm(ref[:512])
    assert np.linalg.norm(C - ref) / np.linalg.norm(ref) <= want
