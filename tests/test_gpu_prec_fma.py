"""TSMM_PREC_FMA: IEEE fma in the working precision for the shapes that the native precision runs on the tensor cores, in
both regimes, aligned and not, alone and in a group."""
import numpy as np
import pytest
import torch

import paper_2208_08088_gb300 as tsmm
import tsmm_inputs as ti
from gpu_util import NP2T, assert_parity, run, to_device

pytestmark = pytest.mark.gpu
FMA = tsmm.PREC_FMA


@pytest.mark.parametrize("pad", [0, 1])
@pytest.mark.parametrize("dtype,m,n,k", [(np.float32, 700, 64, 3000), (np.float32, 261, 20, 40), (np.float64, 1500, 40, 1000),
                                         (np.float32, 300, 200, 24), (np.float32, 300, 200, 100), (np.float64, 200, 130, 40)])
def test_parity_and_chains_of_fmas(dtype, m, n, k, pad):
    for dist in ("uniform", "integer"):
        A, B, C0 = (ti.matrix_np(r, c, s, dist, dtype) for r, c, s in ((m, k, 51), (k, n, 52), (m, n, 53)))
        pb, pl = tsmm.pack_b(to_device(B), precision=FMA), tsmm.plan(m, n, k, NP2T[dtype], FMA)
        C, _, _ = run(A, B, C0, 1.5, 0.5, lda=m + pad, plan=pl, pb=pb)
        assert_parity(C, A, B, C0, 1.5, 0.5, exact=dist == "integer")
    if n <= 64:  # the fma kernel that tsmm_execute_noalloc runs, with the same splits
        dA, dB = to_device(A, ld=m + pad), to_device(B)
        F = tsmm.colmajor(m, n, NP2T[dtype])
        code = tsmm.F32 if dtype == np.float32 else tsmm.F64
        tsmm.tsmm_execute_noalloc(code, m, n, k, 1.0, dA.data_ptr(), m + pad, dB.data_ptr(), k, 0.0, F.data_ptr(), m)
        torch.cuda.synchronize()
        C, _, _ = run(A, B, None, 1.0, 0.0, lda=m + pad, plan=pl, pb=pb)
        np.testing.assert_array_equal(C, F.cpu().numpy())


def test_small_entries_beside_large_ones_keep_their_bits():
    """A row's entries span 2^90, its large ones meet zeros of B: the small products come out as fmas give them."""
    m, n, k = 200, 64, 4096
    rng = np.random.default_rng(41)
    A = np.asfortranarray(rng.uniform(1, 2, (m, k)))
    A[:, 1::2] *= 2.0 ** 90
    B = np.zeros((k, n), order="F")
    B[0, :] = rng.uniform(1, 2, n)
    C, _, _ = run(A, B, None, 1.0, 0.0, plan=tsmm.plan(m, n, k, torch.float64, FMA),
                  pb=tsmm.pack_b(to_device(B), precision=FMA))
    np.testing.assert_array_equal(C, A[:, :1] * B[:1])


def test_groups_mismatches_and_refusals():
    m, n, k = 300, 48, 500
    A, B, _ = (ti.matrix_np(r, c, 54, "uniform", np.float32) for r, c in ((m, k), (k, n), (m, n)))
    dA, dB = to_device(A), to_device(B)
    pb = tsmm.pack_b(dB, precision=FMA)
    outs = [tsmm.colmajor(m, n, torch.float32) for _ in range(2)]
    tsmm.execute(tsmm.plan(m, n, k, torch.float32, FMA), 1.0, dA, pb, 0.0, outs[0])
    native = tsmm.plan(m, n, k, torch.float32)
    tsmm.execute_grouped([(tsmm.plan(m, n, k, torch.float32, FMA), 1.0, dA, pb, 0.0, outs[1])])
    torch.cuda.synchronize()
    assert torch.equal(outs[0], outs[1])
    with pytest.raises(tsmm.TsmmError):
        tsmm.execute(native, 1.0, dA, pb, 0.0, outs[0])
    with pytest.raises(tsmm.TsmmError):
        tsmm.pack_b(dB, precision=3)
