"""The warp-level attention kernel in its two ways of loading keys and values: TMA boxes (pages of 16 tokens, up to 1,024 pages per
sequence) and cp.async (everything else)."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from tests.gpu_harness import make_setup, need_gpu
from workload import configs


def logits_of(hd, page_size, pages, B=3, k=5, P=150):
    """Logits of one verify step of B sequences with k drafts behind P tokens, two layers, heads of hd."""
    b = need_gpu()
    cfg = configs.shrunk(configs.get(1), n_layers=2, vocab=4096, n_docs=200)
    if hd == 128:
        cfg = replace(cfg, model=replace(cfg.model, d_model=512, n_q_heads=4, n_kv_heads=2, head_dim=128, d_ff=1088))
    s = make_setup(replace(cfg, page_size=page_size, prompt_len=P), build_drafter=False, oracle_ngrams=False)
    rng = np.random.default_rng(5)
    tokens = torch.zeros((B, P + 2 * (k + 1)), dtype=torch.int32, device="cuda")
    tokens[:, :P] = torch.from_numpy(rng.integers(0, 4096, (B, P)).astype(np.int32)).cuda()
    drafts = torch.from_numpy(rng.integers(0, 4096, (B, k)).astype(np.int32)).cuda()
    length = torch.tensor([P, P - 37, 2], dtype=torch.int32, device="cuda")
    pool, bt, kv = s.model.new_kv(B, pages * page_size if pages else tokens.shape[1] + b.MAX_ROWS)
    ws = s.model.new_workspace(B, k)
    seqs = b.make_seqs(tokens, length)
    b.tasc_prefill(s.model, kv, seqs, B, P, ws)
    out = b.tasc_verify_step(s.model, kv, seqs, drafts, ws, want_logits=True)[3]
    b.tasc_poll_status(ws)
    return out.cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("hd", [64, 128])
def test_logits_do_not_depend_on_how_keys_are_loaded(hd):
    """Another page size or capacity may split the key ranges differently: float32 sums in another order, and a key or value of the
    second layer on the other side of a bf16 rounding boundary -- the bound of the batch-invariance test, 5e-3."""
    want = logits_of(hd, 16, None)
    for page_size, pages in ((16, 1024), (16, 1025), (8, None), (32, None), (64, 3)):
        got = logits_of(hd, page_size, pages)
        assert np.abs(got - want).max() <= 5e-3, (page_size, pages)


@pytest.mark.gpu
@pytest.mark.parametrize("index,capacity", [(1, 17000), (4, 17000), (4, 8 * 1024 * 16), (4, 8 * 1024 * 16 + 64)])
def test_long_caches_read_by_range(index, capacity):
    """Caches of more pages than a CTA keeps the ids of.  With heads of 128 TMA boxes while each of eight key ranges has no more than 1,024
    pages, cp.async beyond; against pages of 32 tokens, which are never boxes.  (The same ranges and sums: the bound is for the second
    layer's keys.)"""
    b = need_gpu()
    k = 5
    cfg = configs.shrunk(configs.get(index), n_layers=2, vocab=4096, n_docs=200)
    gen = torch.Generator(device="cuda")
    m = cfg.model
    got = []
    for page_size in (16, 32):
        s = make_setup(replace(cfg, page_size=page_size, prompt_len=capacity), build_drafter=False, oracle_ngrams=False)
        gen.manual_seed(3)
        T = capacity // 32 * 32 + 32                                 # tokens of both caches
        kv_tokens = torch.empty((2, 2, 2, T, m.n_kv_heads, m.head_dim), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.5, generator=gen)
        pool, bt, kv = s.model.new_kv(2, capacity)
        pages = bt.shape[1]
        for i in range(2):
            x = kv_tokens[:, :, i, :pages * page_size].reshape(2, 2, pages, page_size, m.n_kv_heads, m.head_dim)
            pool[:, :, bt[i].long()] = x.transpose(3, 4)
        tokens = torch.randint(0, 4096, (2, capacity), generator=gen, device="cuda", dtype=torch.int32)
        drafts = torch.randint(0, 4096, (2, k), generator=gen, device="cuda", dtype=torch.int32)
        length = torch.tensor([capacity - k - 1, capacity // 2], dtype=torch.int32, device="cuda")
        ws = s.model.new_workspace(2, k)
        got.append(b.tasc_verify_step(s.model, kv, b.make_seqs(tokens, length), drafts, ws, want_logits=True)[3].cpu().numpy())
        b.tasc_poll_status(ws)
    assert np.abs(got[0] - got[1]).max() <= 5e-3
