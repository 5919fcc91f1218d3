"""FP32 regime (ii), k > 32, where the last tile's second half of 32 columns lies wholly past column n (n % 64 in
1..32): that half is not stored, and the slots of C that the stores before it still read must not be handed on.  Blocks
walk many items, so every slot is used again.  24-bit integers in A and one nonzero a column in B make every entry of C a
single product plus C0: compared for equality."""
import pytest
import torch

import paper_2208_08088_gb300 as tsmm

pytestmark = pytest.mark.gpu


# a half tile at the end of every wide row of tiles; every second tile a half one
@pytest.mark.parametrize("m,n", [(9984, 7969), (9984, 8016), (600064, 65), (600064, 96)])
@pytest.mark.parametrize("k", [40, 100])  # six slots of C, four
def test_skipped_halves_leave_the_slots_alone(m, n, k):
    g = torch.Generator(device="cuda").manual_seed(2)
    A = tsmm.colmajor(m, k, torch.float32)
    A.copy_(torch.randint(-(2 ** 23) + 1, 2 ** 23, (m, k), generator=g, device="cuda"))
    at = torch.randint(0, k, (n,), generator=g, device="cuda")
    B = tsmm.colmajor(k, n, torch.float32)
    B.zero_()
    B[at, torch.arange(n, device="cuda")] = 1.0
    pb, pl = tsmm.pack_b(B), tsmm.plan(m, n, k, torch.float32)
    C0 = tsmm.colmajor(m, n, torch.float32)
    C0.copy_(torch.randint(-(2 ** 22), 2 ** 22, (m, n), generator=g, device="cuda"))
    C = tsmm.colmajor(m, n, torch.float32)
    for beta in (0.0, 1.0):
        want = A[:, at] + (C0 if beta else 0.0)
        for _ in range(4):
            C.copy_(C0)
            tsmm.execute(pl, 1.0, A, pb, beta, C)
            pl.check()
            assert torch.equal(C, want)
