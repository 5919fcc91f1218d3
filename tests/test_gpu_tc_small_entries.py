"""The FP32 tensor-core kernels on entries that a three-way BF16 split may lose parts of.  An entry too small to matter
leaves every sum on the tensor cores, and a row that needs fmas leaves the others there: the results are those of the same
inputs without that entry or row, bit for bit.  Rows that need them are within the library's bound, however many they are."""
import numpy as np
import pytest

from gpu_util import assert_parity, run

pytestmark = pytest.mark.gpu

SHAPES = [(300, 20, 700), (300, 64, 5000), (261, 48, 64), (300, 200, 50), (300, 97, 128)]  # regime (i), regime (ii)


def draw(m, n, k):
    rng = np.random.default_rng(29)
    A = np.asfortranarray(rng.uniform(-1, 1, (m, k)).astype(np.float32))
    B = np.asfortranarray(rng.uniform(0.5, 1, (k, n)).astype(np.float32))
    return np.abs(A) + np.float32(0.5), B


@pytest.mark.parametrize("m,n,k", SHAPES)
@pytest.mark.parametrize("tiny", [1e-31, 1e-40])
@pytest.mark.parametrize("where", ["a", "b", "both"])
def test_entries_too_small_to_matter(where, tiny, m, n, k):
    A, B = draw(m, n, k)
    out = []
    for v in (0.0, tiny):
        if where in ("a", "both"):
            A[::7, 3] = v
        if where in ("b", "both"):
            B[5, ::3] = v
        out.append(run(A, B, None, 1.0, 0.0)[0])
    np.testing.assert_array_equal(out[0], out[1])


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("count", [1, 4, 16, 17, 128])
@pytest.mark.parametrize("m,n,k", SHAPES)
def test_rows_that_need_fmas(m, n, k, count, pad):
    """`count` rows of the middle slab: infinities, overflows and sums near 2^-120."""
    A, B = draw(m, n, k)
    rows = 128 + np.random.default_rng(31).permutation(128)[:count]
    A[rows[0::3]] *= np.float32(2.0 ** -120)
    A[rows[1::3], k // 2] = np.inf
    A[rows[2::3], k - 1] = np.float32(3e38)
    B[k - 1] *= np.float32(3)
    if count == 1:
        A[rows, 1] = np.nan
    C, _, _ = run(A, B, None, 1.0, 0.0, lda=m + pad)
    with np.errstate(over="ignore", invalid="ignore"):
        ref = (A.astype(np.float64) @ B).astype(np.float32)
    fin = np.isfinite(ref)
    np.testing.assert_array_equal(C[~fin], ref[~fin])
    ok = np.all(fin, axis=1)
    assert_parity(np.asfortranarray(C[ok]), np.asfortranarray(A[ok]), B, None, 1.0, 0.0)
    if count <= 16 or n > 64:
        others = np.setdiff1d(np.arange(m), rows)
        A2 = A.copy(order="F")
        A2[rows] = 1.0
        want = run(A2, B, None, 1.0, 0.0, lda=m + pad)[0]
        np.testing.assert_array_equal(C[others], want[others])
