"""Passes whose decoder layers run as one cooperative kernel (forward_persist.cu): which ones those are, parity at the sizes of its
token blocks, and what its grid barriers and its sums of squares have to guarantee whatever else the GPU does."""
from dataclasses import replace

import numpy as np
import pytest
import torch

from tests.gpu_harness import lockstep, make_setup, need_gpu
from tests.test_gpu_verify import BF16_TOL, check
from workload import configs, corpus, weights as W


def layers_launches(b):
    return b.tasc_launch_counts()["layers"]


def a_step(b, s, host_tokens, drafts_h):
    """A function that runs one verify step from the same committed state and returns its logits, and the workspace."""
    B, P = host_tokens.shape
    k = drafts_h.shape[1]
    tokens = torch.zeros((B, P + 2 * (k + 1)), dtype=torch.int32, device="cuda")
    length0 = torch.full((B,), P, dtype=torch.int32, device="cuda")
    length = length0.clone()
    pool, bt, kv = s.model.new_kv(B, tokens.shape[1] + b.MAX_ROWS)
    ws = s.model.new_workspace(B, k)
    tokens[:, :P] = torch.from_numpy(host_tokens).cuda()
    drafts = torch.from_numpy(drafts_h).cuda()
    seqs = b.make_seqs(tokens, length)
    b.tasc_prefill(s.model, kv, seqs, B, P, ws)
    b.tasc_poll_status(ws)

    def step(keep=(pool, bt, tokens, length, drafts)):
        length.copy_(length0)
        return b.tasc_verify_step(s.model, kv, seqs, drafts, ws, want_logits=True)[3]
    return step, ws


@pytest.mark.gpu
def test_a_kernel_of_another_stream_that_holds_an_sm_is_waited_for():
    """The layers need an SM each to themselves, all at once.  While another stream's kernel holds one for about 1.3 s (longer
    than a barrier's limit within a pass), the step has to wait for it like any other launch: no time-out, same logits."""
    b = need_gpu()
    cfg = configs.shrunk(configs.get(1), n_layers=2, vocab=4096, n_docs=200)
    s = make_setup(cfg, build_drafter=False, oracle_ngrams=False)
    rng = np.random.default_rng(1)
    step, ws = a_step(b, s, rng.integers(0, 4096, (1, 40)).astype(np.int32), rng.integers(0, 4096, (1, 5)).astype(np.int32))
    before = layers_launches(b)
    want = step().cpu().numpy()
    assert layers_launches(b) == before + 1
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        torch.cuda._sleep(2_500_000_000)
    got = step()
    b.tasc_poll_status(ws)
    assert np.array_equal(got.cpu().numpy(), want)


@pytest.mark.gpu
@pytest.mark.parametrize("B,k", [(1, 5), (4, 3), (8, 5)])
def test_sums_of_squares_do_not_depend_on_the_order_of_the_ctas(B, k):
    """A residual row whose squares make any change of the order of the additions visible: one feature's square is a^2 in
    [2^24, 2^25), one 1 (the middle between two floats), the other hundreds are 2^-34.  Added behind a^2 in double a CTA's few of
    these vanish, among themselves they do not, and a^2 + 1 then rounds to the next float instead of back to a^2.  (The residual
    projections are zero, so the row stays what it is.)  The step's logits must be the same bits every time -- and for the same
    row times a power of two, which reaches every part of the sum's range, as long as the squares do not overflow."""
    b = need_gpu()
    cfg = configs.shrunk(configs.get(1), n_layers=4, vocab=512, n_docs=200)
    d = cfg.model.d_model
    f32 = np.float32

    def factor(ss):
        return f32(1) / np.sqrt(f32(f32(ss) * f32(f32(1) / f32(d)) + f32(cfg.model.rms_eps)))
    a = next(v for v in range(4096, 5760, 32) if factor(v * v) != factor(v * v + 2))
    w = W.make_weights(cfg.model, 0, gain_jitter=0.1)
    row = np.full(d, 2.0 ** -17, dtype=f32)
    row[:12] = 0.0
    row[0], row[5] = a, 1.0
    w["lm_head"] = w["lm_head"].copy()
    for layer in w["layers"]:
        layer["wo"] = np.zeros_like(layer["wo"])
        layer["w_down"] = np.zeros_like(layer["w_down"])
    rng = np.random.default_rng(2)
    prompts, drafts = rng.integers(0, 512, (B, 3)).astype(np.int32), rng.integers(0, 512, (B, k)).astype(np.int32)
    want = None
    for power in (0, 7, 23, 40, 56):
        w["embed"] = np.tile(row * f32(2.0) ** power, (cfg.model.vocab, 1))
        s = make_setup(cfg, build_drafter=False, oracle_ngrams=False, host_w=w)
        step, ws = a_step(b, s, prompts, drafts)
        before = layers_launches(b)
        first = step().clone()
        assert layers_launches(b) == before + 1
        different = sum(int(not torch.equal(step(), first)) for _ in range(40))
        b.tasc_poll_status(ws)
        assert different == 0, f"2^{power}: {different} of 40 repetitions differ"
        want = first if want is None else want
        assert bool((first == 0).all()) if power == 56 else torch.equal(first, want), f"2^{power}"


def shape_of(hd, n_layers):
    """Configuration 1's shape, or one with heads of 128."""
    cfg = configs.shrunk(configs.get(1), n_layers=n_layers, vocab=4096, n_docs=500)
    if hd == 128:
        cfg = replace(cfg, model=replace(cfg.model, d_model=512, n_q_heads=4, n_kv_heads=2, head_dim=128, d_ff=1088))
    return cfg


@pytest.mark.gpu
@pytest.mark.parametrize("hd", [64, 128])
@pytest.mark.parametrize("B,k,P", [(11, 2, 40), (5, 6, 130), (8, 5, 200), (7, 8, 33), (16, 3, 70)])
def test_two_blocks_of_32_rows(B, k, P, hd):
    """33, 35, 48, 63 and 64 rows: a second block of token rows with one row, some, or all of them in use.  Two layers; the oracle
    runs the first, a middle and the last sequence."""
    b = need_gpu()
    cfg = replace(shape_of(hd, 2), prompt_len=P)
    s = make_setup(cfg)
    prompts = corpus.make_prompts(cfg, B, prompt_len=P)
    before = layers_launches(b)
    rep = lockstep(s, prompts, k + 3, k, oracle_rows=sorted({0, B // 2, B - 1}), **BF16_TOL)
    assert layers_launches(b) - before >= rep.steps
    check(rep, f"two blocks of 32 rows, heads of {hd}, B={B} k={k} P={P}")


@pytest.mark.gpu
@pytest.mark.parametrize("which,B,k,P,one", [(1, 1, 1, 20, 1), (1, 2, 7, 20, 1), (1, 3, 5, 20, 0), (1, 8, 3, 20, 0), (1, 11, 2, 20, 1), (1, 16, 3, 20, 1),
                                             (1, 13, 4, 20, 0), (2, 2, 3, 20, 1), (2, 3, 2, 20, 0), (4, 1, 6, 3030, 1), (4, 1, 6, 3100, 0)])
def test_which_steps_run_their_layers_as_one_kernel(which, B, k, P, one):
    """2, 16, 18, 32, 33, 64 and 65 rows of the small layers, 8 and 9 of larger ones, and heads of 128 with 12 key ranges of 256 and
    of more keys."""
    b = need_gpu()
    cfg = replace(configs.shrunk(configs.get(which), n_layers=1, vocab=512, n_docs=100), prompt_len=P)
    s = make_setup(cfg, build_drafter=False, oracle_ngrams=False)
    rng = np.random.default_rng(3)
    step, ws = a_step(b, s, rng.integers(0, 512, (B, P)).astype(np.int32), rng.integers(0, 512, (B, k)).astype(np.int32))
    before = layers_launches(b)
    step()
    b.tasc_poll_status(ws)
    assert layers_launches(b) - before == one


@pytest.mark.gpu
@pytest.mark.parametrize("B,k", [(1, 5), (4, 3), (7, 8)])
def test_a_step_is_bitwise_repeatable(B, k):
    """6, 16 and 63 rows behind 300 tokens, four layers: split key ranges and their merge included."""
    b = need_gpu()
    s = make_setup(shape_of(64, 4), build_drafter=False, oracle_ngrams=False)
    rng = np.random.default_rng(4)
    step, ws = a_step(b, s, rng.integers(0, 4096, (B, 300)).astype(np.int32), rng.integers(0, 4096, (B, k)).astype(np.int32))
    before = layers_launches(b)
    want = step().clone()
    assert layers_launches(b) == before + 1
    for _ in range(10):
        assert torch.equal(step(), want)
    b.tasc_poll_status(ws)


@pytest.mark.gpu
@pytest.mark.parametrize("B,k", [(2, 5), (7, 6)])
def test_generate_graph_replay_equals_plain_enqueue(B, k):
    """tasc_generate with its step replayed from a graph (a side stream) and enqueued (the default stream), steps of 12 and 49
    rows: the same tokens and statistics."""
    b = need_gpu()
    cfg = shape_of(64, 4)
    s = make_setup(cfg, oracle_ngrams=False)
    max_new = 30
    prompts = corpus.make_prompts(cfg, B, prompt_len=100)
    results = []
    for side in (False, True):
        tokens = torch.zeros((B, 100 + max_new + k + 2), dtype=torch.int32, device="cuda")
        tokens[:, :100] = torch.from_numpy(prompts).cuda()
        length = torch.full((B,), 100, dtype=torch.int32, device="cuda")
        pool, bt, kv = s.model.new_kv(B, tokens.shape[1] + b.MAX_ROWS)
        ws = s.model.new_workspace(B, k)
        stream = torch.cuda.Stream() if side else torch.cuda.current_stream()
        stream.wait_stream(torch.cuda.current_stream())
        before = layers_launches(b)
        with torch.cuda.stream(stream):
            out, st = b.tasc_generate(s.model, s.drafter, kv, b.make_seqs(tokens, length), B, max_new, k, ws)
        torch.cuda.current_stream().wait_stream(stream)
        assert layers_launches(b) > before
        results.append((out.cpu().numpy(), st.steps, list(st.accepted_hist)))
    assert np.array_equal(results[0][0], results[1][0])
    assert results[0][1:] == results[1][1:]
