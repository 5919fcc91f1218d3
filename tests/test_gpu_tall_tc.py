"""FP32 regime (i) with n > 16 on the tensor cores (exact three-way BF16 splits): every MMA width, edges of slabs and
chunks, and the inputs that a split cannot carry, which the block recomputes with plain fmas.  Tolerances: the
library's componentwise bound, or equality where every partial sum is exactly representable."""
import numpy as np
import pytest
import torch

import paper_2208_08088_gb300 as tsmm
import tsmm_inputs as ti
from gpu_util import assert_parity, run, to_device

pytestmark = pytest.mark.gpu


def gen(m, n, k, dist="uniform"):
    return tuple(ti.matrix_np(r, c, s, dist, np.float32) for r, c, s in ((m, k, 21), (k, n, 22), (m, n, 23)))


@pytest.mark.parametrize("n", [17, 32, 33, 48, 49, 64])
@pytest.mark.parametrize("m,k,pad", [(1, 1, 0), (127, 31, 1), (128, 32, 0), (129, 33, 3), (260, 97, 0), (2305, 4100, 3)])
def test_widths_and_edges(m, n, k, pad):
    A, B, C0 = gen(m, n, k)
    C, pl, _ = run(A, B, C0, -1.25, 0.75, lda=m + pad)
    assert pl.info()["bm"] == 128
    assert_parity(C, A, B, C0, -1.25, 0.75)
    A, B, C0 = gen(m, n, k, "integer")
    C, _, _ = run(A, B, C0, 1.5, 0.5, lda=m + pad)
    assert_parity(C, A, B, C0, 1.5, 0.5, exact=True)


@pytest.mark.parametrize("dtype,n,m,k0", [(np.float32, 20, 261, 28), (np.float64, 20, 7000, 256)])
@pytest.mark.parametrize("dk", [0, 3, 4, 5, 7, 8, 31, 33])  # whole chunks of k by tensor copies, the rest column by column
@pytest.mark.parametrize("offset,pad", [(0, 1), (0, 2), (1, 0), (2, 3), (3, 1)])
def test_unaligned_columns(dtype, n, m, k0, dk, offset, pad):
    """A in NaNs, its columns at every offset from 16 bytes: nothing beside them is used, the last chunk is complete."""
    k = k0 + dk
    A, B, C0 = (ti.matrix_np(r, c, s, "integer", dtype) for r, c, s in ((m, k, 21), (k, n, 22), (m, n, 23)))
    C, pl, _ = run(A, B, C0, 1.0, 1.0, lda=m + pad, a_offset=offset)
    assert pl.info()["bm"] == 128
    assert_parity(C, A, B, C0, 1.0, 1.0, exact=True)


@pytest.mark.parametrize("lda", [264, 265])  # tensor copies; columns moved one by one
@pytest.mark.parametrize("n", [24, 40, 64])
def test_wide_integers_are_exact(n, lda):
    """24-bit entries fill all three pieces; B has one nonzero a column, so C is a single product, exact."""
    m, k = 264, 200
    rng = np.random.default_rng(3)
    A = np.asfortranarray(rng.integers(-(2 ** 24) + 1, 2 ** 24, size=(m, k)).astype(np.float32))
    B = np.zeros((k, n), np.float32, order="F")
    B[rng.integers(0, k, n), np.arange(n)] = 1.0
    C, _, _ = run(A, B, None, 1.0, 0.0, lda=lda)
    np.testing.assert_array_equal(C, (A.astype(np.float64) @ B).astype(np.float32))


@pytest.mark.parametrize("lda", [300, 301])
@pytest.mark.parametrize("k", [70, 5000])  # one split; several
@pytest.mark.parametrize("what", ["inf_a", "nan_a", "inf_b", "overflow", "tiny", "tiny_b", "huge"])
@pytest.mark.parametrize("n", [20, 64])
def test_values_a_split_cannot_carry(what, n, k, lda):
    m = 300
    A, B, C0 = (x.copy(order="F") for x in gen(m, n, k, "integer"))
    exact = True
    if what == "inf_a":
        A[140, k - 1] = np.inf
    elif what == "nan_a":
        A[7, 3] = np.nan
    elif what == "inf_b":
        B[k // 2, n - 1] = -np.inf
    elif what == "overflow":  # the products overflow, the entries do not (one sign: infinite in any order)
        A[200, :] = 3e38
        B = np.abs(B) + np.float32(1)
    elif what == "huge":  # rounds to infinity as BF16, finite as FP32
        A[299, 5] = np.finfo(np.float32).max
        B[5, :] = 0.5
        exact = False
    elif what == "tiny":  # products of 2^-130, sums exact subnormals
        A *= np.float32(2.0 ** -70)
        B *= np.float32(2.0 ** -60)
        C0 *= np.float32(2.0 ** -130)
    else:  # some columns subnormal, others not
        B[:, ::3] *= np.float32(2.0 ** -140)
        C0[:, ::3] *= np.float32(2.0 ** -140)
    C, _, _ = run(A, B, C0, 1.0, 1.0, lda=lda)
    if what == "overflow":  # the oracle's FP64 sums stay finite: infinite once rounded to FP32, the other rows exact
        ref = (A.astype(np.float64) @ B + C0).astype(np.float32)
        assert np.all(np.isposinf(ref[200]))
        np.testing.assert_array_equal(C, ref)
        return
    assert_parity(C, A, B, C0, 1.0, 1.0, exact=exact and what in ("tiny", "tiny_b"))


def test_grouped_widths_equal_single_launches():
    """Problems of all three MMA widths, aligned and not, with specials in one: bit for bit the single launches."""
    items, single, outs = [], [], []
    for i, (m, n, k, pad) in enumerate([(500, 17, 300, 0), (1000, 32, 2000, 1), (129, 40, 64, 3), (700, 48, 999, 0),
                                        (2000, 64, 3000, 0), (333, 63, 5000, 2), (64, 16, 128, 0)]):
        A, B, C0 = gen(m, n, k)
        if i == 3:
            A[5, 5] = np.inf
        dA, pb = to_device(A, ld=m + pad), tsmm.pack_b(to_device(B))
        c1, c2 = to_device(C0), to_device(C0)
        p1, p2 = tsmm.plan(m, n, k, torch.float32), tsmm.plan(m, n, k, torch.float32)
        tsmm.execute(p1, 1.5, dA, pb, 0.5, c1)
        items.append((p2, 1.5, dA, pb, 0.5, c2))
        single.append((p1, c1))
        outs.append(c2)
    tsmm.execute_grouped(items)
    for (p1, c1), (p2, *_), c2 in zip(single, items, outs):
        p1.check()
        p2.check()
        np.testing.assert_array_equal(c1.cpu().numpy(), c2.cpu().numpy())
