"""FP64 regime (i) on the tensor cores (exact digit products, k >= 256, n > 1): every MMA width, edges of slabs and
steps, rows whose scale grows within an item, and the inputs the digits cannot carry, which the block recomputes with
FP64 fmas.  Tolerances: the library's componentwise bound against the Dot2 oracle, or equality where every partial sum is
exactly representable."""
import numpy as np
import pytest
import torch

import paper_2208_08088_gb300 as tsmm
from gpu_util import assert_parity, run, to_device

pytestmark = pytest.mark.gpu


def gen(m, n, k, dist="uniform"):
    rng = np.random.default_rng(31)
    draw = (lambda r, c: rng.uniform(-1, 1, (c, r)).T) if dist == "uniform" else \
        (lambda r, c: rng.integers(-4, 5, (c, r)).astype(np.float64).T)
    return draw(m, k), draw(k, n), draw(m, n)


def rows_for(n, k, extra):
    """The fewest rows that the digits serve (m * padded n * k >= 4e7), and a few more."""
    np_ = next(w for w in (2, 4, 8, 16, 24, 32, 48, 64) if w >= n)
    return -(-40_000_000 // (np_ * k)) + extra


@pytest.mark.parametrize("n", [2, 15, 17, 33, 48, 64])
@pytest.mark.parametrize("extra,k,pad", [(0, 256, 0), (1, 257, 1), (63, 319, 0), (130, 1025, 3), (5, 4100, 1)])
def test_widths_and_edges(extra, n, k, pad):
    m = rows_for(n, k, extra)
    A, B, C0 = gen(m, n, k)
    C, pl, _ = run(A, B, C0, -1.25, 0.75, lda=m + pad)
    assert pl.info()["bm"] == 128
    assert_parity(C, A, B, C0, -1.25, 0.75)
    A, B, C0 = gen(m, n, k, "integer")
    C, _, _ = run(A, B, C0, 1.5, 0.5, lda=m + pad)
    assert_parity(C, A, B, C0, 1.5, 0.5, exact=True)


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("n", [4, 30, 64])
def test_growing_rows_are_exact(n, pad):
    """Entries grow along k by powers of two, at other places in every row: scales grow in mid-group, sums are shifted.
    Integers below 2^21 against integers below 16: every sum exact."""
    k = 900
    m = rows_for(n, k, 6) // 2 * 2
    lda = m + pad
    rng = np.random.default_rng(5)
    A = rng.integers(-8, 9, size=(m, k)).astype(np.float64)
    for i in range(m):
        for p in rng.integers(0, k, size=6):
            A[i, p:] *= 8.0
    A = np.asfortranarray(A)
    B = np.asfortranarray(rng.integers(1, 16, size=(k, n)).astype(np.float64))
    C, _, _ = run(A, B, None, 1.0, 0.0, lda=lda)
    np.testing.assert_array_equal(C, A @ B)


@pytest.mark.parametrize("n", [3, 20, 64])
@pytest.mark.parametrize("dist", ["normal", "lognormal", "sparse", "identity", "zero_rows", "triangular"])
def test_distributions_within_bound(dist, n):
    """What the guard proves and what it hands to the fmas (single products stay exact: identity)."""
    k = 700
    m = rows_for(n, k, 3)
    rng = np.random.default_rng(8)
    A = rng.standard_normal((m, k))
    B = rng.standard_normal((k, n))
    if dist == "lognormal":
        A, B = np.exp(6 * A), np.exp(6 * B)
    elif dist == "sparse":
        A *= rng.random((m, k)) < 0.01
        B *= rng.random((k, n)) < 0.05
    elif dist == "identity":
        A *= np.exp2(rng.integers(-30, 30, size=(m, k)).astype(np.float64))
        B = np.zeros((k, n))
        B[rng.integers(0, k, n), np.arange(n)] = 1.0
    elif dist == "zero_rows":
        A[::3] = 0.0
        B[:, 0] = 0.0
    elif dist == "triangular":
        A *= np.arange(k)[None, :] >= 2 * (np.arange(m)[:, None] % 350)
    A, B = np.asfortranarray(A), np.asfortranarray(B)
    C, _, _ = run(A, B, None, 1.0, 0.0)
    if dist == "identity":
        np.testing.assert_array_equal(C, A @ B)
    assert_parity(C, A, B, None, 1.0, 0.0)


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("what", ["inf_a", "nan_a", "inf_b", "huge", "tiny_a", "tiny_b", "subnormal"])
@pytest.mark.parametrize("n,k", [(5, 700), (64, 5000)])
def test_values_the_digits_cannot_carry(what, n, k, pad):
    m = rows_for(n, k, 300) // 2 * 2
    lda = m + pad
    A, B, C0 = (x.copy(order="F") for x in gen(m, n, k, "integer"))
    if what == "inf_a":
        A[140, k - 1] = np.inf
    elif what == "nan_a":
        A[7, 3] = np.nan
    elif what == "inf_b":
        B[k // 2, n - 1] = -np.inf
    elif what == "huge":
        A[200, 5] = 1e300
    elif what == "tiny_a":
        A[:130] *= 1e-200
    elif what == "tiny_b":
        B[:, ::3] *= 1e-200
    else:
        A[17] *= 5e-324
        C0[17] = 0.0
    exact = what == "subnormal"
    C, _, _ = run(A, B, C0, 1.0, 1.0, lda=lda)
    assert_parity(C, A, B, C0, 1.0, 1.0, exact=exact)


def test_grouped_widths_equal_single_launches():
    items, single, outs = [], [], []
    for i, (m, n, k, pad) in enumerate([(9000, 2, 3000, 0), (1300, 16, 2000, 1), (3300, 40, 256, 1), (900, 48, 999, 0),
                                        (2000, 64, 3000, 0), (333, 63, 5000, 1), (64, 16, 128, 0), (200, 1, 900, 0)]):
        A, B, C0 = gen(m, n, k)
        if i == 3:
            A[5, 5] = np.inf
        dA, pb = to_device(A, ld=m + pad), tsmm.pack_b(to_device(B))
        c1, c2 = to_device(C0), to_device(C0)
        p1, p2 = tsmm.plan(m, n, k, torch.float64), tsmm.plan(m, n, k, torch.float64)
        tsmm.execute(p1, 1.5, dA, pb, 0.5, c1)
        items.append((p2, 1.5, dA, pb, 0.5, c2))
        single.append((p1, c1))
        outs.append(c2)
    tsmm.execute_grouped(items)
    for (p1, c1), (p2, *_), c2 in zip(single, items, outs):
        p1.check()
        p2.check()
        np.testing.assert_array_equal(c1.cpu().numpy(), c2.cpu().numpy())
