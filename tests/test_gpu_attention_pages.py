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
