"""Passes of 33 to 96 rows of the small layers in token tiles of 16 rows: against the one-kernel layers (33 to 64 rows, caches of up to
352 tokens) and against the same sequences alone.  The bound is the batch-invariance test's, 5e-3: float32 sums in another order, keys
and values of later layers on the other side of a bf16 rounding boundary."""
import numpy as np
import pytest
import torch

from tests.gpu_harness import make_setup, need_gpu
from tests.test_gpu_one_kernel_layers import layers_launches, shape_of


def step_logits(b, s, tokens_h, drafts_h, capacity):
    """Logits of one verify step behind the given tokens, and whether its layers were one kernel."""
    B, P = tokens_h.shape
    k = drafts_h.shape[1]
    tokens = torch.zeros((B, P + 2 * (k + 1)), dtype=torch.int32, device="cuda")
    tokens[:, :P] = torch.from_numpy(tokens_h).cuda()
    length = torch.full((B,), P, dtype=torch.int32, device="cuda")
    pool, bt, kv = s.model.new_kv(B, capacity)
    ws = s.model.new_workspace(B, k)
    seqs = b.make_seqs(tokens, length)
    b.tasc_prefill(s.model, kv, seqs, B, P, ws)
    before = layers_launches(b)
    out = b.tasc_verify_step(s.model, kv, seqs, torch.from_numpy(drafts_h).cuda(), ws, want_logits=True)[3]
    b.tasc_poll_status(ws)
    return out.cpu().numpy(), layers_launches(b) - before


@pytest.mark.gpu
@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("B,k", [(11, 2), (5, 6), (8, 5), (16, 3)])
def test_kernels_per_phase_agree_with_one_kernel(B, k, hd):
    """33, 35, 48 and 64 rows."""
    b = need_gpu()
    s = make_setup(shape_of(hd, 2), build_drafter=False, oracle_ngrams=False)
    rng = np.random.default_rng(B)
    tokens, drafts = rng.integers(0, 4096, (B, 90)).astype(np.int32), rng.integers(0, 4096, (B, k)).astype(np.int32)
    want, one = step_logits(b, s, tokens, drafts, 352)
    got, none = step_logits(b, s, tokens, drafts, 353)
    assert (one, none) == (1, 0)
    assert np.abs(got - want).max() <= 5e-3


@pytest.mark.gpu
@pytest.mark.parametrize("B,k", [(13, 4), (19, 3), (12, 7), (16, 5), (49, 1)])
def test_a_sequence_does_not_depend_on_its_batch(B, k):
    """65, 76, 96 (8 and 6 to a sequence) and 98 rows, the last in tiles of 32: the first, a middle and the last sequence alone."""
    b = need_gpu()
    s = make_setup(shape_of(64, 2), build_drafter=False, oracle_ngrams=False)
    rng = np.random.default_rng(B)
    tokens, drafts = rng.integers(0, 4096, (B, 70)).astype(np.int32), rng.integers(0, 4096, (B, k)).astype(np.int32)
    all_, _ = step_logits(b, s, tokens, drafts, 112)
    for i in (0, B // 2, B - 1):
        alone, _ = step_logits(b, s, tokens[i:i + 1], drafts[i:i + 1], 112)
        assert np.abs(all_[i] - alone[0]).max() <= 5e-3, i
