"""Attention whose key ranges are split over a cluster: rows go straight into the merging CTA's shared memory where that leaves as many CTAs
to an SM, otherwise they are fetched.  Query rows that do not divide by the splits, ranges without keys, sequences without rows, both
ways of handing rows over, 32-, 64- and 128-wide heads; the oracle runs the first and the last sequence."""
from dataclasses import replace

import pytest

from tests.gpu_harness import lockstep, make_setup
from tests.test_gpu_verify import BF16_TOL, check
from workload import configs, corpus


@pytest.mark.gpu
@pytest.mark.parametrize("hd,n_q,n_kv,B,k,P", [
    (64, 9, 3, 11, 8, 900),         # 27 rows per KV head
    (64, 14, 2, 9, 3, 700),         # 28 rows
    (64, 14, 2, 3, 8, 300),         # 63 rows
    (128, 12, 2, 4, 2, 1500),       # 18 rows, heads in one CTA
    (128, 12, 2, 2, 6, 900),        # heads of one KV head dealt out to several CTAs
    (128, 12, 2, 6, 8, 700),        # 54 rows: fetched
    (32, 8, 2, 10, 1, 500),         # 8 rows, fewer than some clusters have CTAs
    (32, 16, 2, 5, 7, 40),          # a range for every tile, some without keys
])
def test_split_key_ranges(hd, n_q, n_kv, B, k, P):
    base = configs.shrunk(configs.get(2), n_layers=2, vocab=4096, n_docs=500, d_ff=1024)
    cfg = replace(base, model=replace(base.model, d_model=n_q * hd, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=hd), prompt_len=P)
    s = make_setup(cfg)
    rep = lockstep(s, corpus.make_prompts(cfg, B, prompt_len=P), k + 3, k, oracle_rows=sorted({0, B - 1}), **BF16_TOL)
    check(rep, f"split key ranges, heads of {hd}, {n_q} / {n_kv}, B={B} k={k} P={P}")
