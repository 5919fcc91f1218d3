"""FP64 regime (i) on the tensor cores against the fma chain: on data whose rows or columns are unevenly scaled, the error
(2-norm, against compensated sums) is no larger than that of the FP64 fma kernel, which tsmm_execute_noalloc runs, on the
same inputs."""
import numpy as np
import pytest
import torch

import oracle
import paper_2208_08088_gb300 as tsmm
from gpu_util import to_device

pytestmark = pytest.mark.gpu


def draw(dist, m, n, k):
    rng = np.random.default_rng(17)
    A, B = rng.standard_normal((m, k)), rng.standard_normal((k, n))
    if dist == "rows":  # every row of A and of B at its own size
        A, B = A * 10.0 ** rng.uniform(-3, 3, (m, 1)), B * 10.0 ** rng.uniform(-3, 3, (k, 1))
    elif dist == "inverse":  # columns of A against rows of B
        u = rng.uniform(-2, 2, k)
        A, B = A * np.exp2(u), B * np.exp2(-u)[:, None]
    return np.asfortranarray(A), np.asfortranarray(B)


@pytest.mark.parametrize("dist", ["normal", "rows", "inverse"])
@pytest.mark.parametrize("k", [2048, 8192])
@pytest.mark.parametrize("n", [16, 40, 49, 64])
def test_error_is_no_larger_than_the_fma_chains(n, k, dist):
    m = max(260, -(-40_000_000 // ({16: 16, 40: 48}.get(n, 64) * k)))
    A, B = draw(dist, m, n, k)
    dA, dB = to_device(A), to_device(B)
    C = {}
    pb, pl = tsmm.pack_b(dB), tsmm.plan(m, n, k, torch.float64)
    assert pl.info()["bm"] == 128
    for which in ("digits", "fma"):
        out = tsmm.colmajor(m, n, torch.float64)
        if which == "digits":
            tsmm.execute(pl, 1.0, dA, pb, 0.0, out)
            pl.check()
        else:
            tsmm.tsmm_execute_noalloc(tsmm.F64, m, n, k, 1.0, dA.data_ptr(), m, dB.data_ptr(), k, 0.0, out.data_ptr(), m)
            torch.cuda.synchronize()
        C[which] = out.cpu().numpy()[:260]
    ref, _ = oracle.tsmm(1.0, np.asfortranarray(A[:260]), B, 0.0, None)
    err = {w: np.linalg.norm(c - ref) / np.linalg.norm(ref) for w, c in C.items()}
    assert err["digits"] <= err["fma"], err
