"""FP32 regime (ii) with k > 32 on the tensor cores (exact three-way BF16 splits): edges of tiles and chunks, both forms
of C, blocks that walk many items, and the inputs that a split cannot carry, which the epilogue recomputes with plain
fmas.  Tolerances: the library's componentwise bound, or equality where every partial sum is exactly representable."""
import numpy as np
import pytest
import torch

import paper_2208_08088_gb300 as tsmm
import tsmm_inputs as ti
from gpu_util import assert_parity, run, to_device

pytestmark = pytest.mark.gpu


def gen(m, n, k, dist="uniform"):
    return tuple(ti.matrix_np(r, c, s, dist, np.float32) for r, c, s in ((m, k, 41), (k, n, 42), (m, n, 43)))


# (pad of lda, pad of ldc): C by tensor copies; by element; A through the aligned scratch
@pytest.mark.parametrize("pa,pc", [(0, 0), (0, 1), (1, 0)])
@pytest.mark.parametrize("k", [33, 48, 64, 65, 97, 128])
@pytest.mark.parametrize("m,n", [(4, 65), (128, 96), (132, 128), (516, 417)])
def test_edges(m, n, k, pa, pc):
    A, B, C0 = gen(m, n, k)
    for alpha, beta in ((1.0, 0.0), (1.0, 1.0), (-1.25, 0.75)):
        C, _, _ = run(A, B, C0, alpha, beta, lda=m + pa, ldc=m + pc)
        assert_parity(C, A, B, C0, alpha, beta)
    A, B, C0 = gen(m, n, k, "integer")
    C, _, _ = run(A, B, C0, 1.5, 0.5, lda=m + pa, ldc=m + pc)
    assert_parity(C, A, B, C0, 1.5, 0.5, exact=True)


@pytest.mark.parametrize("k", [40, 100])
@pytest.mark.parametrize("ldc", [9984, 9985])
def test_wide_integers_over_many_items(k, ldc):
    """24-bit entries fill all three pieces; B has one nonzero a column, so C is a single product plus C0, exact.  Every
    block walks several items of several tiles, slots and rings wrap."""
    m, n = 9984, 8000
    g = torch.Generator(device="cuda").manual_seed(1)
    A = tsmm.colmajor(m, k, torch.float32)
    A.copy_(torch.randint(-(2 ** 23) + 1, 2 ** 23, (m, k), generator=g, device="cuda"))
    at = torch.randint(0, k, (n,), generator=g, device="cuda")
    B = tsmm.colmajor(k, n, torch.float32)
    B.zero_()
    B[at, torch.arange(n, device="cuda")] = 1.0
    pb, pl = tsmm.pack_b(B), tsmm.plan(m, n, k, torch.float32)
    for beta in (0.0, 1.0):
        C = tsmm.colmajor(m, n, torch.float32, ld=ldc)
        C.copy_(torch.randint(-(2 ** 22), 2 ** 22, (m, n), generator=g, device="cuda"))
        want = A[:, at] + (C if beta else 0.0)
        tsmm.execute(pl, 1.0, A, pb, beta, C)
        pl.check()
        assert torch.equal(C, want)


@pytest.mark.parametrize("ldc", [300, 301])
@pytest.mark.parametrize("k", [50, 128])
@pytest.mark.parametrize("what", ["inf_a", "nan_a", "inf_b", "overflow", "tiny", "tiny_b", "huge"])
def test_values_a_split_cannot_carry(what, k, ldc):
    m, n = 300, 200
    A, B, C0 = (x.copy(order="F") for x in gen(m, n, k, "integer"))
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
    elif what == "tiny":  # products of 2^-130, sums exact subnormals
        A *= np.float32(2.0 ** -70)
        B *= np.float32(2.0 ** -60)
        C0 *= np.float32(2.0 ** -130)
    else:  # some columns subnormal, others not
        B[:, ::3] *= np.float32(2.0 ** -140)
        C0[:, ::3] *= np.float32(2.0 ** -140)
    C, _, _ = run(A, B, C0, 1.0, 1.0, ldc=ldc)
    if what == "overflow":  # the oracle's FP64 sums stay finite: infinite once rounded to FP32, the other rows exact
        ref = (A.astype(np.float64) @ B + C0).astype(np.float32)
        assert np.all(np.isposinf(ref[200]))
        np.testing.assert_array_equal(C, ref)
        return
    assert_parity(C, A, B, C0, 1.0, 1.0, exact=what in ("tiny", "tiny_b"))


def test_beta_zero_ignores_c():
    m, n, k = 260, 300, 70
    A, B, _ = gen(m, n, k)
    pb, pl = tsmm.pack_b(to_device(B)), tsmm.plan(m, n, k, torch.float32)
    for ldc in (m, m + 1):
        C = to_device(np.full((m, n), np.nan, np.float32), ld=ldc)
        tsmm.execute(pl, 2.0, to_device(A), pb, 0.0, C)
        pl.check()
        assert_parity(C.cpu().numpy(), A, B, None, 2.0, 0.0)
