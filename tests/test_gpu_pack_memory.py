"""A B whose packed panel fits the memory that is left, and whose tensor-core form beside it does not: accepted, packed
without that form, and multiplied by the fma kernels, alone and in a group."""
import pytest
import torch

import paper_2208_08088_gb300 as tsmm

pytestmark = pytest.mark.gpu


def ints(r, c, dtype, gen):
    M = tsmm.colmajor(r, c, dtype)
    M.copy_(torch.randint(-1, 2, (r, c), generator=gen, device="cuda"))
    return M


@pytest.mark.parametrize("dtype,k,left", [(torch.float32, 1 << 22, 1700 << 20), (torch.float64, 1 << 20, 1200 << 20)])
def test_panel_alone_when_memory_is_short(dtype, k, left):
    m, n = 40, 64
    gen = torch.Generator(device="cuda").manual_seed(3)
    A, B = ints(m, k, dtype, gen), ints(k, n, dtype, gen)
    want = (A.double() @ B.double()).to(dtype)
    small = tsmm.pack_b(ints(256, n, dtype, gen))  # its kernels are loaded before the memory is taken
    plans = [tsmm.plan(m, n, k, dtype) for _ in range(2)]
    outs = [tsmm.colmajor(m, n, dtype) for _ in range(3)]
    tsmm.execute(tsmm.plan(m, n, 256, dtype), 1.0, A[:, :256], small, 0.0, outs[2])
    tsmm.tsmm_execute_noalloc(tsmm.F64 if dtype == torch.float64 else tsmm.F32, m, n, 256, 1.0, A.data_ptr(), m, B.data_ptr(),
                              k, 0.0, outs[2].data_ptr(), m)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    taken = torch.empty(torch.cuda.mem_get_info()[0] - left, dtype=torch.uint8, device="cuda")
    try:
        before = torch.cuda.mem_get_info()[0]
        pb = tsmm.pack_b(B)
        used = before - torch.cuda.mem_get_info()[0]
        assert used < 1.25 * pb.info()["bytes"]  # the panel alone
        tsmm.execute(plans[0], 1.0, A, pb, 0.0, outs[0])
        tsmm.execute_grouped([(plans[1], 1.0, A, pb, 0.0, outs[1]), (plans[0], 1.0, A, pb, 0.0, outs[2])])
        torch.cuda.synchronize()
        plans[0].check()
        equal = [torch.equal(o, want) for o in outs]
    finally:
        del taken
        torch.cuda.empty_cache()
    assert all(equal)
    # the same plan with a B that has its form again
    pb2 = tsmm.pack_b(B)
    outs[0].zero_()
    tsmm.execute(plans[0], 1.0, A, pb2, 0.0, outs[0])
    tsmm.execute(plans[0], 1.0, A, pb, 0.0, outs[1])
    plans[0].check()
    assert torch.equal(outs[0], want) and torch.equal(outs[1], want)
