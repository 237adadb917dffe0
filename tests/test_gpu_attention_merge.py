"""Attention whose key ranges are split over a cluster: rows go straight into the merging CTA's shared memory where that leaves room for as many
clusters, otherwise they are fetched.  Query rows that do not divide by the splits, fewer rows than splits, ranges without keys, sequences without
rows, prompts of different lengths, both kernels and both ways of handing rows over, 32-, 64- and 128-wide heads; the oracle runs the first and the last
sequence.  Which kernel and which way a case takes is looked at: the rules that choose them may change."""
from dataclasses import replace

import numpy as np
import pytest

from tests.gpu_harness import attention_of_steps, lockstep, make_setup, need_gpu
from tests.test_gpu_verify import BF16_TOL, check
from workload import configs, corpus

PUSHED, FETCHED, WHOLE = "pushed", "fetched", "one key range"


@pytest.mark.gpu
@pytest.mark.parametrize("hd,n_q,n_kv,B,k,P,page,spare,tcgen05,way", [
    (64, 9, 3, 11, 8, 900, 16, 0, False, PUSHED),       # 27 rows per KV head
    (64, 14, 2, 9, 3, 700, 16, 0, False, PUSHED),       # 28 rows
    (64, 14, 2, 3, 8, 300, 16, 0, False, PUSHED),       # 63 rows
    (64, 14, 2, 4, 8, 900, 8, 0, False, PUSHED),        # pages that are not TMA boxes
    (128, 12, 2, 4, 2, 1500, 16, 0, False, PUSHED),     # 18 rows, heads in one CTA
    (128, 12, 2, 2, 6, 900, 16, 0, False, PUSHED),      # heads of one KV head dealt out to several CTAs
    (128, 12, 2, 6, 8, 700, 8, 0, False, FETCHED),      # 54 rows of 128-wide heads: no room behind the ring
    (128, 12, 2, 6, 8, 90, 8, 650, False, FETCHED),     # the same, ranges without keys
    (128, 12, 2, 6, 8, 700, 16, 0, True, PUSHED),
    (128, 12, 2, 6, 8, 90, 16, 650, True, PUSHED),      # ranges without keys
    (64, 2, 2, 9, 1, 900, 16, 0, False, PUSHED),        # two rows, fewer than the clusters have CTAs
    (32, 8, 2, 2, 1, 900, 16, 0, False, PUSHED),        # 8 rows
    (32, 16, 2, 2, 7, 600, 16, 0, False, PUSHED),       # 64 rows of 32-wide heads: two CTAs per SM with and without them
    (32, 16, 2, 2, 7, 40, 16, 600, False, PUSHED),      # ranges without keys
    (32, 8, 2, 10, 1, 500, 16, 0, False, WHOLE),
    (32, 16, 2, 5, 7, 40, 16, 0, False, WHOLE),
])
def test_split_key_ranges(hd, n_q, n_kv, B, k, P, page, spare, tcgen05, way, monkeypatch):
    base = configs.shrunk(configs.get(2), n_layers=2, vocab=4096, n_docs=500, d_ff=1024)
    cfg = replace(base, model=replace(base.model, d_model=n_q * hd, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=hd), prompt_len=P + spare, page_size=page)
    plans = attention_of_steps(need_gpu(), monkeypatch)
    s = make_setup(cfg)
    lengths = np.linspace(P, max(2, P * 2 // 3), B).astype(int)
    rep = lockstep(s, corpus.make_prompts(cfg, B, prompt_len=P), k + 3, k, oracle_rows=sorted({0, B - 1}), lengths=lengths, spare=spare, **BF16_TOL)
    check(rep, f"split key ranges, heads of {hd}, {n_q} / {n_kv}, B={B} k={k} P={P}")
    for p in plans:
        assert p["tcgen05"] == tcgen05 and (p["splits"] == 1) == (way == WHOLE) and (p["push_rows"] > 0) == (way == PUSHED), plans
        if spare:
            assert p["splits"] * 64 > P + 64                                          # more ranges than the keys make tiles
