"""A sequence whose token buffer is longer than its cache, by more pages than a CTA of any attention kernel keeps the ids of (1,024 pages
of 16 tokens in one key range): the call reports ENOKV, the sequences beside it and the calls behind it are what they are without it."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from tests.gpu_harness import make_setup, need_gpu
from workload import configs

LONG = 20000


def model_of(index):
    cfg = configs.shrunk(configs.get(index), n_layers=2, vocab=4096, n_docs=200)
    return make_setup(replace(cfg, prompt_len=LONG), build_drafter=False, oracle_ngrams=False)


# the one-kernel layers, the warp-level attention, the tcgen05 attention: all keys of a sequence are one CTA's
@pytest.mark.gpu
@pytest.mark.parametrize("index,B,k,capacity", [(1, 1, 5, 112), (1, 5, 4, 112), (4, 64, 6, 1552)])
def test_a_sequence_longer_than_its_cache(index, B, k, capacity):
    b = need_gpu()
    s = model_of(index)
    rng = np.random.default_rng(index + B)
    P = 60
    tokens = torch.from_numpy(rng.integers(0, 4096, (B, LONG + 2 * (k + 1))).astype(np.int32)).cuda()
    drafts = torch.from_numpy(rng.integers(0, 4096, (B, k)).astype(np.int32)).cuda()
    length = torch.full((B,), P, dtype=torch.int32, device="cuda")
    pool, bt, kv = s.model.new_kv(B, capacity)
    ws = s.model.new_workspace(B, k)
    seqs = b.make_seqs(tokens, length)
    keep = tokens.clone()

    def step(first):
        tokens.copy_(keep)
        length.fill_(P)
        length[0] = first
        return b.tasc_verify_step(s.model, kv, seqs, drafts, ws, want_logits=True)[3].view(B, k + 1, -1).cpu().numpy()

    b.tasc_prefill(s.model, kv, seqs, B, P, ws)
    want = step(P)
    b.tasc_poll_status(ws)
    for first in (LONG, 16 * 1024 + 1, 16 * 1025):
        got = step(first)
        with pytest.raises(b.TascError) as e:
            b.tasc_poll_status(ws)
        assert e.value.code == b.ENOKV
        assert np.array_equal(got[1:], want[1:])
    assert np.array_equal(step(P), want)
    b.tasc_poll_status(ws)


@pytest.mark.gpu
@pytest.mark.parametrize("index", [1, 4])
def test_a_prompt_longer_than_its_cache(index):
    b = need_gpu()
    s = model_of(index)
    rng = np.random.default_rng(index)
    tokens = torch.from_numpy(rng.integers(0, 4096, (2, LONG + 4)).astype(np.int32)).cuda()
    length = torch.tensor([LONG, 60], dtype=torch.int32, device="cuda")
    pool, bt, kv = s.model.new_kv(2, 112)
    ws = s.model.new_workspace(2, 1)
    b.tasc_prefill(s.model, kv, b.make_seqs(tokens, length), 2, LONG, ws)
    with pytest.raises(b.TascError) as e:
        b.tasc_poll_status(ws)
    assert e.value.code == b.ENOKV
    got = pool.clone()
    length[0] = 100
    b.tasc_prefill(s.model, kv, b.make_seqs(tokens, length), 2, 100, ws)
    b.tasc_poll_status(ws)
    # (another launch shape: keys and values of the second layer may be on the other side of a bf16 rounding boundary)
    err = (pool.float() - got.float()).abs().max() / pool.float().abs().max()
    assert float(err) <= 2 ** -7
