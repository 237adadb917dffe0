"""The device memory that the set-up calls keep for the next one, and the call that gives it back."""
import pytest
import torch

from tests.gpu_harness import need_gpu


@pytest.mark.gpu
def test_what_the_set_up_calls_keep_is_given_back():
    """Corpus tables of 16 M windows take a block of about half a gigabyte.  It stays with the library (no more than 2 GB) until
    tasc_scratch_release, which leaves the drafter that is alive as it is."""
    b = need_gpu()
    n = 1 << 24
    tokens = torch.randint(0, 50000, (n,), dtype=torch.int32, device="cuda")
    contexts, length = tokens[:256].view(1, 256).contiguous(), torch.tensor([200], dtype=torch.int32, device="cuda")

    def free():
        return torch.cuda.mem_get_info()[0]

    def build_and_draft(n):
        drafter = b.tasc_drafter_build(tokens[:n], torch.tensor([0, n], dtype=torch.int64, device="cuda"), 2, 2, 50000)
        return drafter, b.tasc_draft(drafter, contexts, length, 4)
    small, drafts = build_and_draft(1000)                  # (all code that runs below is loaded, the pool is made)
    del small
    b.tasc_scratch_release()
    before = free()
    drafter, drafts = build_and_draft(n)
    torch.cuda.synchronize()
    kept = before - free()
    assert 300e6 < kept < 2.2e9
    b.tasc_scratch_release()
    assert before - free() < 128e6                         # the drafter's tables
    assert b.tasc_draft(drafter, contexts, length, 4).tolist() == drafts.tolist()
    del drafter
    b.tasc_scratch_release()
    assert before - free() < 40e6
