"""FP64 regime (ii) with k >= 4 on the tensor cores (exact digit products): edges of tiles and chunks of k, both forms of C,
blocks that walk tiles of several rows of A, and the outputs that the digits cannot carry, which the epilogue recomputes
with FP64 fmas (few rows of a warp, and all).  Tolerances: the library's componentwise bound against the Dot2 oracle, or
equality where every partial sum is exactly representable."""
import numpy as np
import pytest
import torch

import paper_2208_08088_gb300 as tsmm
from gpu_util import assert_parity, run, to_device

pytestmark = pytest.mark.gpu


def gen(m, n, k, dist="uniform"):
    rng = np.random.default_rng(37)
    draw = (lambda r, c: rng.uniform(-1, 1, (c, r)).T) if dist == "uniform" else \
        (lambda r, c: rng.integers(-4, 5, (c, r)).astype(np.float64).T)
    return draw(m, k), draw(k, n), draw(m, n)


@pytest.mark.parametrize("pad", [0, 1])  # C by tensor copies; by element
@pytest.mark.parametrize("k", [3, 4, 15, 32, 33, 64, 65, 97, 128])
@pytest.mark.parametrize("m,n", [(2, 65), (128, 80), (130, 129), (514, 417)])
def test_edges(m, n, k, pad):
    A, B, C0 = gen(m, n, k)
    for alpha, beta in ((1.0, 0.0), (1.0, 1.0), (-1.25, 0.75)):
        C, _, _ = run(A, B, C0, alpha, beta, lda=m + pad, ldc=m + pad)
        assert_parity(C, A, B, C0, alpha, beta)
    A, B, C0 = gen(m, n, k, "integer")
    C, _, _ = run(A, B, C0, 1.5, 0.5, lda=m + pad, ldc=m + pad)
    assert_parity(C, A, B, C0, 1.5, 0.5, exact=True)


@pytest.mark.parametrize("k", [20, 60, 90, 128])
@pytest.mark.parametrize("ldc", [4984, 4985])
def test_wide_integers_over_many_tiles(k, ldc):
    """52-bit entries against one nonzero a column: C is a single product plus C0, exact.  Every block walks many tiles and
    crosses rows of A; slots and rings wrap."""
    m, n = 4984, 3000
    g = torch.Generator(device="cuda").manual_seed(1)
    A = tsmm.colmajor(m, k, torch.float64)
    A.copy_(torch.randint(-(2 ** 51) + 1, 2 ** 51, (m, k), generator=g, device="cuda"))
    at = torch.randint(0, k, (n,), generator=g, device="cuda")
    B = tsmm.colmajor(k, n, torch.float64)
    B.zero_()
    B[at, torch.arange(n, device="cuda")] = 1.0
    pb, pl = tsmm.pack_b(B), tsmm.plan(m, n, k, torch.float64)
    for beta in (0.0, 1.0):
        C = tsmm.colmajor(m, n, torch.float64, ld=ldc)
        C.copy_(torch.randint(-(2 ** 51), 2 ** 51, (m, n), generator=g, device="cuda"))
        want = A[:, at] + (C if beta else 0.0)
        tsmm.execute(pl, 1.0, A, pb, beta, C)
        pl.check()
        assert torch.equal(C, want)


@pytest.mark.parametrize("k", [24, 128])
def test_exact_sums(k):
    """Integers whose sums fill the significand, of either sign and with cancellation: exact in any order."""
    m, n = 260, 200
    rng = np.random.default_rng(3)
    A = np.asfortranarray(rng.integers(-(2 ** 31), 2 ** 31, (m, k)).astype(np.float64))
    B = np.asfortranarray(rng.integers(-(2 ** 14), 2 ** 14, (k, n)).astype(np.float64))
    B[:, ::3] = np.where(np.arange(k)[:, None] % 2 == 0, 1.0, -1.0)
    A[:, 1::2] = A[:, ::2] + rng.integers(-3, 4, (m, k // 2))
    C, _, _ = run(A, B, None, 1.0, 0.0)
    np.testing.assert_array_equal(C, A @ B)


@pytest.mark.parametrize("ldc", [300, 301])
@pytest.mark.parametrize("k", [10, 50, 128])
@pytest.mark.parametrize("what", ["inf_a", "nan_a", "inf_b", "zero_rows_inf_b", "overflow", "tiny", "huge", "sparse",
                                  "few_uneven_rows", "uneven_rows"])
def test_outputs_the_digits_cannot_carry(what, k, ldc):
    m, n = 300, 200
    A, B, C0 = (x.copy(order="F") for x in gen(m, n, k))
    rng = np.random.default_rng(9)
    if what == "inf_a":
        A[140, k - 1] = np.inf
    elif what == "nan_a":
        A[7, 3] = np.nan
    elif what in ("inf_b", "zero_rows_inf_b"):
        B[k // 2, n - 1] = -np.inf
        if what != "inf_b":
            A[:200] = 0.0
    elif what == "overflow":  # the products overflow, the entries do not (one sign: infinite in any order)
        A[200, :] = 1e300
        B = np.abs(B) * 1e9 + 1e9
    elif what == "tiny":
        A *= 2.0 ** -500
        C0 *= 2.0 ** -500
    elif what == "huge":
        A[:, ::2] *= 2.0 ** 500
        C0 *= 2.0 ** 500
    elif what == "sparse":
        A *= rng.random((m, k)) < 0.15
        B *= rng.random((k, n)) < 0.15
    else:  # rows whose large entry meets a zero of B: the others lie 2^-40 below the row's scale
        rows = [3, 77, 290] if what == "few_uneven_rows" else slice(None)
        A[rows] *= 2.0 ** -40
        A[rows, 0] = 1.0
        B[0, ::2] = 0.0
    C, _, _ = run(A, B, C0, 1.0, 1.0, ldc=ldc)
    if what == "overflow":
        assert np.all(np.isposinf(C[200]))
        keep = np.arange(m) != 200
        C, A, C0 = (np.asfortranarray(x[keep]) for x in (C, A, C0))
        assert_parity(C, A, B, C0, 1.0, 1.0)
        return
    assert_parity(C, A, B, C0, 1.0, 1.0)


def test_beta_zero_ignores_c():
    m, n, k = 260, 300, 40
    A, B, _ = gen(m, n, k)
    pb, pl = tsmm.pack_b(to_device(B)), tsmm.plan(m, n, k, torch.float64)
    for ldc in (m, m + 1):
        C = to_device(np.full((m, n), np.nan), ld=ldc)
        tsmm.execute(pl, 2.0, to_device(A), pb, 0.0, C)
        pl.check()
        assert_parity(C.cpu().numpy(), A, B, None, 2.0, 0.0)
