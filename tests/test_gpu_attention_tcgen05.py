"""The tcgen05 attention: query tiles of up to 64 and up to 128 rows, 64- and 128-wide heads, contexts that end just before, at and just behind
a tile of 128 keys, one key range and several, ranges of one, two and more tiles (the two places of S and P, and of O, are used in turn), tiles of 64
keys, prompts of one length and of different ones; the oracle runs the first and the last sequence.  That a case takes this kernel is looked at."""
from dataclasses import replace

import pytest

from tests.gpu_harness import attention_of_steps, lockstep, make_setup, need_gpu
from tests.test_gpu_verify import BF16_TOL, check
from workload import configs, corpus


@pytest.mark.gpu
@pytest.mark.parametrize("hd,n_q,n_kv,B,k,P,split,spare", [
    (64, 14, 2, 34, 8, 127, False, 150),        # 63 rows
    (64, 14, 2, 34, 7, 128, False, 150),        # 56 rows
    (64, 16, 2, 34, 7, 249, False, 0),          # 64 rows: a full tile
    (64, 16, 2, 34, 8, 250, False, 0),          # 72 rows: the wider one
    (64, 16, 2, 20, 15, 385, True, 0),          # 128 rows
    (128, 12, 2, 48, 4, 600, False, 0),         # 30 rows
    (128, 12, 2, 66, 6, 260, False, 0),         # 42 rows
    (128, 12, 2, 30, 8, 700, True, 0),          # 54 rows, split
    (128, 16, 2, 34, 8, 383, False, 0),         # 72 rows
    (128, 16, 2, 24, 15, 640, True, 0),         # 128 rows
])
@pytest.mark.parametrize("ragged", [False, True])
def test_tiles_and_key_ranges(hd, n_q, n_kv, B, k, P, split, spare, ragged, monkeypatch):
    base = configs.shrunk(configs.get(2), n_layers=2, vocab=4096, n_docs=500, d_ff=1024)
    cfg = replace(base, model=replace(base.model, d_model=n_q * hd, n_q_heads=n_q, n_kv_heads=n_kv, head_dim=hd), prompt_len=P + spare)
    plans = attention_of_steps(need_gpu(), monkeypatch)
    s = make_setup(cfg)
    lengths = [P - i * (P // 2) // B for i in range(B)] if ragged else None
    rep = lockstep(s, corpus.make_prompts(cfg, B, prompt_len=P), k + 3, k, oracle_rows=sorted({0, B - 1}), lengths=lengths, spare=spare, **BF16_TOL)
    check(rep, f"tcgen05 attention, heads of {hd}, {n_q} / {n_kv}, B={B} k={k} P={P}")
    for p in plans:
        assert p["tcgen05"] and (p["splits"] > 1) == split, plans


@pytest.mark.gpu
@pytest.mark.parametrize("hd,B,P,tile,split", [(128, 3, 49, 64, False)] + [(hd, 3, P, 64 if P < 68 else 128, False) for hd in (64, 128) for P in (64, 65, 67, 84, 100, 128, 130, 260)]
                         + [(hd, 1, P, 64, True) for hd in (64, 128) for P in (150, 190, 193)])
def test_prompts_in_tiles_of_64_and_128_keys(hd, B, P, tile, split, monkeypatch):
    """Blocks of 16 prompt tokens and 8 query heads are 128 rows: tiles of 64 keys where one or two of them hold all keys, and in several ranges."""
    b, k = need_gpu(), 2
    base = configs.shrunk(configs.get(2), n_layers=2, vocab=4096, n_docs=500, d_ff=1024)
    cfg = replace(base, model=replace(base.model, d_model=16 * hd, n_q_heads=16, n_kv_heads=2, head_dim=hd), prompt_len=P)
    plans, prefill = [], b.tasc_prefill

    def watched(model, kv, *args):
        plans.append(b.tasc_attention_plan(model, kv, B, (P + 14) // 16 * 16))
        before = b.tasc_launch_counts()["attention_split"]
        prefill(model, kv, *args)
        assert b.tasc_launch_counts()["attention_split"] - before == model.shape.n_layers

    monkeypatch.setattr(b, "tasc_prefill", watched)
    s = make_setup(cfg)
    rep = lockstep(s, corpus.make_prompts(cfg, B, prompt_len=P), 2, k, oracle_rows=sorted({0, B - 1}), lengths=[P, P // 2, P - 5][:B], spare=-16, **BF16_TOL)
    check(rep, f"tcgen05 attention, prompts of {P}, heads of {hd}")
    assert [(p["tcgen05"], p["tile"], p["splits"] > 1) for p in plans] == [(True, tile, split)]
