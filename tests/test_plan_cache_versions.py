"""Plan-cache files from before the tensor-core kernels: their split counts are kept and written back as such, but not
forced on plans whose kernel has other stages and slabs."""
import os

import pytest
import torch

import paper_2208_08088_gb300 as tsmm

OLD = "# tsmm plan cache v2: dtype m n k sm_count splits\n"
NEW = "# tsmm plan cache v3\n"


@pytest.fixture(autouse=True)
def empty_cache():
    tsmm.tsmm_plan_cache_clear()
    yield
    tsmm.tsmm_plan_cache_clear()


def sections(path):
    """The file's entries under its two marks."""
    out, at = {"v2": [], "v3": []}, None
    for line in path.read_text().splitlines():
        if line.startswith("# tsmm plan cache v"):
            at = line.split()[4].rstrip(":")
        elif line and not line.startswith("#"):
            out[at].append(line)
    return out


def test_entries_keep_their_version(tmp_path):
    src, dst, again = (tmp_path / n for n in ("a", "b", "c"))
    src.write_text("f32 4096 64 4096 152 5\n" + NEW + "f32 4096 48 4096 152 3\n" + OLD + "f64 4096 8 4096 152 2\n")
    tsmm.tsmm_plan_cache_load(str(src))
    tsmm.tsmm_plan_cache_save(str(dst))
    want = {"v2": ["f32 4096 64 4096 152 5", "f64 4096 8 4096 152 2"], "v3": ["f32 4096 48 4096 152 3"]}
    assert sections(dst) == want
    tsmm.tsmm_plan_cache_clear()
    tsmm.tsmm_plan_cache_load(str(dst))
    tsmm.tsmm_plan_cache_save(str(again))
    assert sections(again) == want


def test_an_old_entry_does_not_replace_a_new_one(tmp_path):
    new, old, dst = (tmp_path / n for n in ("a", "b", "c"))
    new.write_text(NEW + "f32 4096 64 4096 152 5\nf32 4096 16 4096 152 5\n")
    old.write_text(OLD + "f32 4096 64 4096 152 7\nf32 4096 16 4096 152 7\n")
    for path in (new, old):
        tsmm.tsmm_plan_cache_load(str(path))
    tsmm.tsmm_plan_cache_save(str(dst))
    assert sections(dst) == {"v2": ["f32 4096 16 4096 152 7"], "v3": ["f32 4096 64 4096 152 5"]}


@pytest.mark.gpu
@pytest.mark.parametrize("m,n,k,dtype,tensor", [(4096, 64, 4096, torch.float32, True), (4096, 8, 4096, torch.float64, True),
                                                (4096, 16, 4096, torch.float32, False), (64, 8, 4096, torch.float64, False)])
def test_old_counts_are_not_forced_on_tensor_core_plans(m, n, k, dtype, tensor, tmp_path):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    name = "f64" if dtype == torch.float64 else "f32"
    chosen = tsmm.plan(m, n, k, dtype).info()["splits"]
    forced = 2 if chosen != 2 else 4
    path = tmp_path / "cache"
    for mark, used in ((OLD, not tensor), ("", not tensor), (NEW, True)):
        path.write_text(f"{mark}{name} {m} {n} {k} {sms} {forced}\n")
        tsmm.tsmm_plan_cache_clear()
        tsmm.tsmm_plan_cache_load(os.fspath(path))
        assert tsmm.plan(m, n, k, dtype).info()["splits"] == (forced if used else chosen)
