"""The framework's work in use, as cases that can be timed: what a program that serves one task on one GPU calls.

Kinds of case
  step       one speculative step of a batch: tasc_draft, then tasc_verify_step (what a serving loop calls per step)
  prefill    tasc_prefill of a batch of prompts
  generate   tasc_generate of a batch: prefill, then speculative steps until every sequence has its new tokens
  task       a task's set-up from its output corpus: statistics, corpus tables, and the first drafts made with them
  tokenizer  vocabulary enrichment: added tokens chosen on a sample of the corpus, their embedding rows, the corpus re-encoded

Models, corpus recipes, draft lengths and context lengths are those of the repository's configurations (workload/configs.py);
"0.5b-merged" is configuration 3's shape (the 0.5B decoder with 8,192 added tokens).  All inputs are random, made on the GPU
from the seed.
"""
from __future__ import annotations

import math
from dataclasses import replace

import torch

from paper_2602_24174_b200 import binding as b
from workload import configs

# name -> (configuration, largest batch of a step, largest context of a step)
MODELS = {
    "tiny-f32": (0, 8, 96),
    "135m": (1, 32, 512),
    "0.5b": (2, 32, 1024),
    "0.5b-merged": (3, 32, 1024),
    "1.5b": (4, 64, 1536),
}


def listed():
    return [
        # the smallest call there is: configuration 0, the float32 decoder, one sequence
        {"name": "step tiny-f32 B=1", "kind": "step", "model": "tiny-f32", "batch": 1, "k": 4, "ctx": 64, "ragged": False},
        # one user talking to the smallest bf16 model: latency
        {"name": "step 135m B=1", "kind": "step", "model": "135m", "batch": 1, "k": 5, "ctx": 270, "ragged": False},
        # the small model serving its configuration's batch, sequences of different lengths
        {"name": "step 135m B=16", "kind": "step", "model": "135m", "batch": 16, "k": 5, "ctx": 380, "ragged": True},
        # a handful of users, an odd batch and short drafts
        {"name": "step 0.5b B=7", "kind": "step", "model": "0.5b", "batch": 7, "k": 3, "ctx": 560, "ragged": True},
        # the enlarged vocabulary at the widest draft, a full batch (288 rows)
        {"name": "step 0.5b-merged B=32", "kind": "step", "model": "0.5b-merged", "batch": 32, "k": 8, "ctx": 640, "ragged": True},
        # the headline: the largest model, one sequence, behind its 1,024-token prompt
        {"name": "step 1.5b B=1", "kind": "step", "model": "1.5b", "batch": 1, "k": 6, "ctx": 1071, "ragged": False},
        # the largest model at its configuration's largest batch, contexts all over the range of a generation
        {"name": "step 1.5b B=64", "kind": "step", "model": "1.5b", "batch": 64, "k": 6, "ctx": 1530, "ragged": True},
        # time to the first token of one short prompt
        {"name": "prefill 135m B=1", "kind": "prefill", "model": "135m", "batch": 1, "ctx": 256, "ragged": False},
        # a batch of long ragged prompts arriving together (the largest case)
        {"name": "prefill 1.5b B=16", "kind": "prefill", "model": "1.5b", "batch": 16, "ctx": 1024, "ragged": True},
        # a whole request batch through one call: prefill and decode, targets from held-out text (teacher-forced)
        {"name": "generate 0.5b B=8", "kind": "generate", "model": "0.5b", "batch": 8, "k": 5, "ctx": 512, "ragged": True, "new": 64},
        # configuration 2's corpus: 200,000 documents, 14 M tokens
        {"name": "task 200k docs", "kind": "task", "recipe": 2, "docs": 200000},
        # enrichment of the 0.5B vocabulary on a 20,000-document sample, then 100,000 documents re-encoded
        {"name": "tokenizer 20k docs", "kind": "tokenizer", "recipe": 2, "docs": 20000, "encode_docs": 100000, "budget": 256, "n_max": 4},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choices(("step", "prefill", "generate", "task", "tokenizer"), weights=(7, 2, 1, 1, 1))[0]
    if kind == "task":
        return {"kind": kind, "recipe": rng.choice((1, 2)), "docs": _log_int(rng, 2000, 200000)}
    if kind == "tokenizer":
        docs = _log_int(rng, 1000, 20000)
        return {"kind": kind, "recipe": rng.choice((1, 2)), "docs": docs, "encode_docs": docs * rng.randint(1, 5),
                "budget": _log_int(rng, 16, 256), "n_max": rng.randint(2, 5)}
    if kind == "step":
        name = rng.choice(("tiny-f32", "135m", "135m", "0.5b", "0.5b", "0.5b-merged", "1.5b", "1.5b"))
        index, b_max, ctx_max = MODELS[name]
        return {"kind": kind, "model": name, "batch": _log_int(rng, 1, b_max), "k": rng.randint(3, 8),
                "ctx": _log_int(rng, 32 if index == 0 else 100, ctx_max), "ragged": rng.random() < 0.6}
    name = rng.choice(("135m", "0.5b", "1.5b"))
    if kind == "prefill":
        return {"kind": kind, "model": name, "batch": _log_int(rng, 1, 16), "ctx": _log_int(rng, 48, 1024), "ragged": rng.random() < 0.6}
    # (the generation of a 1.5B batch would cost more than the largest listed case: fewer sequences and tokens there)
    big = name == "1.5b"
    return {"kind": kind, "model": name, "batch": _log_int(rng, 1, 4 if big else 16), "k": rng.randint(3, 8),
            "ctx": _log_int(rng, 64, 512), "ragged": rng.random() < 0.6, "new": rng.randint(8, 24 if big else 64)}


# ------------------------------------------------------------------------------------------------------------ inputs
def _shape(name):
    cfg = configs.get(MODELS[name][0])
    m = cfg.model
    return replace(m, vocab=m.vocab + cfg.n_merged_tokens), cfg


def _corpus(recipe, vocab, n_docs, gen):
    """A task corpus by the configurations' recipe (documents = phrases drawn by Zipf rank from a fixed pool, uniform
    random tokens inserted at a fixed rate), as (tokens int32[T], offsets int64[n_docs + 1]) on the GPU."""
    dev = "cuda"
    ri = lambda lo, hi, *shape: torch.randint(lo, hi, shape, generator=gen, device=dev)
    n = recipe.pool_size
    plen = ri(recipe.phrase_lo, recipe.phrase_hi + 1, n)
    poff = torch.zeros(n + 1, dtype=torch.int64, device=dev)
    poff[1:] = plen.cumsum(0)
    ptok = ri(0, vocab, n * recipe.phrase_hi)
    w = torch.arange(1, n + 1, dtype=torch.float64, device=dev) ** (-recipe.zipf_s)
    cdf = (w / w.sum()).cumsum(0)
    hi = recipe.len_hi
    max_ph = -(-hi // recipe.phrase_lo)
    toks, lens = [], []
    for d0 in range(0, n_docs, 25000):
        D = min(25000, n_docs - d0)
        ln = ri(recipe.len_lo, recipe.len_hi + 1, D)
        ins = torch.rand((D, hi), generator=gen, device=dev) < recipe.insert_rate
        rank = torch.searchsorted(cdf, torch.rand((D, max_ph), generator=gen, device=dev, dtype=torch.float64)).clamp_(max=n - 1)
        ends = plen[rank].cumsum(1)                                   # phrase boundaries of each document's phrase stream
        src = (~ins).cumsum(1) - (~ins).long()                        # stream position consumed at each output position
        which = torch.searchsorted(ends, src, right=True).clamp_(max=max_ph - 1)
        within = src - (ends - plen[rank]).gather(1, which)
        tok = ptok[poff[rank.gather(1, which)] + within]
        tok = torch.where(ins, ri(0, vocab, D, hi), tok)
        toks.append(tok[torch.arange(hi, device=dev)[None, :] < ln[:, None]].to(torch.int32))
        lens.append(ln)
    off = torch.zeros(n_docs + 1, dtype=torch.int64, device=dev)
    off[1:] = torch.cat(lens).cumsum(0)
    return torch.cat(toks).contiguous(), off


def _text(recipe, vocab, rows, length, gen):
    """Prompts or held-out text that reads like the corpus: documents one after another, cut to [rows, length]."""
    n_docs = rows * length // recipe.len_lo + 2
    return _corpus(recipe, vocab, n_docs, gen)[0][:rows * length].view(rows, length).contiguous()


def _weights(s, gen):
    """Random weights of a decoder shape.  Matrices N(0, 0.02), residual projections scaled by 1 / sqrt(2 L) and tied
    embeddings of 0.1, so that the residual stream and the logits have the spread of a trained model (a top token that
    stands out) instead of the near ties of unscaled random weights."""
    td = torch.float32 if s.dtype == "f32" else torch.bfloat16
    dev = "cuda"

    def mat(rows, cols, std=0.02):
        return torch.empty((rows, cols), dtype=td, device=dev).normal_(0.0, std, generator=gen)

    def gain():
        return torch.empty(s.d_model, device=dev).normal_(1.0, 0.1, generator=gen)

    out = 0.02 / math.sqrt(2 * s.n_layers)
    w = {"embed": mat(s.vocab, s.d_model, 0.1), "final_norm": gain(), "layers": []}
    w["lm_head"] = w["embed"]
    for _ in range(s.n_layers):
        w["layers"].append({"attn_norm": gain(), "wqkv": mat(s.qkv_rows, s.d_model), "wo": mat(s.d_model, s.q_dim, out),
                            "mlp_norm": gain(), "w_gate_up": mat(2 * s.d_ff, s.d_model), "w_down": mat(s.d_model, s.d_ff, out)})
    return w


def _lengths(case, gen):
    """Committed tokens of every sequence: `ctx`, or anything from half of it up to it."""
    B, ctx = case["batch"], case["ctx"]
    if not case["ragged"]:
        return torch.full((B,), ctx, dtype=torch.int32, device="cuda")
    n = torch.randint(max(2, ctx // 2), ctx + 1, (B,), generator=gen, device="cuda", dtype=torch.int32)
    n[0] = ctx
    return n


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    st = {"case": case}
    kind = case["kind"]
    if kind in ("task", "tokenizer"):
        cfg = configs.get(case["recipe"])
        st["cfg"] = cfg
        V = cfg.model.vocab
        if kind == "task":
            st["corpus"] = _corpus(cfg.corpus, V, case["docs"], gen)
            st["tokens"] = _text(cfg.corpus, V, 256, 128, gen)        # contexts that will be drafted for
            st["length"] = torch.randint(64, 129, (256,), generator=gen, device="cuda", dtype=torch.int32)
        else:
            tokens, off = _corpus(cfg.corpus, V, case["encode_docs"], gen)
            st["corpus"] = (tokens, off)
            off_s = off[:case["docs"] + 1].contiguous()
            st["sample"] = (tokens[:int(off_s[-1])].contiguous(), off_s)
            st["embed"] = torch.empty((V, cfg.model.d_model), dtype=torch.bfloat16, device="cuda").normal_(0.0, 0.1, generator=gen)
        return st
    s, cfg = _shape(case["model"])
    B, k = case["batch"], case.get("k", 1)
    new = case.get("new", 0)
    stride = case["ctx"] + new + 2 * (k + 1)
    st["cfg"] = cfg
    st["model"] = b.Model(s, _weights(s, gen), max_positions=stride + b.MAX_ROWS, page_size=cfg.page_size)
    st["workspace"] = st["model"].new_workspace(B, k)
    st["pool"], st["block_table"], st["kv"] = st["model"].new_kv(B, stride + b.MAX_ROWS)
    st["tokens"] = torch.zeros((B, stride), dtype=torch.int32, device="cuda")
    st["tokens"][:, :case["ctx"]] = _text(cfg.corpus, s.vocab, B, case["ctx"], gen)
    st["length0"] = _lengths(case, gen)
    st["length"] = st["length0"].clone()
    st["seqs"] = b.make_seqs(st["tokens"], st["length"])
    if kind != "prefill":
        docs = _corpus(cfg.corpus, s.vocab, min(cfg.corpus.n_docs, 20000), gen)
        st["drafter"] = b.tasc_drafter_build(*docs, cfg.n_max, cfg.p_min, s.vocab)
    if kind == "step":
        # the cache of the committed tokens: K and V of unit-scale inputs through N(0, 0.02) projections
        st["pool"].normal_(0.0, 0.02 * math.sqrt(s.d_model), generator=gen)
        st["drafts"] = torch.empty((B, k), dtype=torch.int32, device="cuda")
    if kind == "generate":
        st["continuation"] = _text(cfg.corpus, s.vocab, B, new + k + 1, gen)
        st["stream"] = torch.cuda.Stream()
    return st


# ------------------------------------------------------------------------------------------------------------ passes
def run(st):
    case, kind = st["case"], st["case"]["kind"]
    if kind == "step":
        st["length"].copy_(st["length0"])                              # the scheduler's view of the batch
        cfg = st["cfg"]
        drafts = b.tasc_draft(st["drafter"], st["tokens"], st["length"], case["k"], cfg.lambda_num, cfg.lambda_den, out=st["drafts"])
        n_acc, nxt, tgt, _ = b.tasc_verify_step(st["model"], st["kv"], st["seqs"], drafts, st["workspace"], want_targets=True)
        return {"drafts": drafts, "accepted": n_acc, "next": nxt, "targets": tgt, "tokens": st["tokens"], "length": st["length"],
                "kv": st["pool"]}
    if kind == "prefill":
        b.tasc_prefill(st["model"], st["kv"], st["seqs"], case["batch"], case["ctx"], st["workspace"])
        return {"kv": st["pool"]}
    if kind == "generate":
        # not on the default stream: the loop then replays a CUDA graph
        st["stream"].wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(st["stream"]):
            st["length"].copy_(st["length0"])
            out, stats = b.tasc_generate(st["model"], st["drafter"], st["kv"], st["seqs"], case["batch"], case["new"], case["k"],
                                         st["workspace"], mode=b.MODE_CONTINUATION, continuation=st["continuation"])
        torch.cuda.current_stream().wait_stream(st["stream"])
        return {"out": out, "steps": stats.steps, "accepted": list(stats.accepted_hist), "tokens": st["tokens"], "length": st["length"],
                "kv": st["pool"]}
    cfg = st["cfg"]
    if kind == "task":
        stats = b.tasc_corpus_stats(*st["corpus"], cfg.model.vocab)
        drafter = b.tasc_drafter_build(*st["corpus"], cfg.n_max, cfg.p_min, cfg.model.vocab)
        drafts = b.tasc_draft(drafter, st["tokens"], st["length"], cfg.k, cfg.lambda_num, cfg.lambda_den)
        return {"statistics": stats, "drafts": drafts}
    merges, sample, sample_off = b.tasc_tok_enrich(*st["sample"], cfg.model.vocab, case["budget"], case["n_max"])
    rows = b.tasc_tok_init_rows(st["embed"], merges)
    tokens, off = b.tasc_tok_encode(*st["corpus"], cfg.model.vocab, merges)
    # into buffers of a fixed size, as a program keeps them whose corpora differ in length
    hi = cfg.corpus.len_hi
    sample = torch.nn.functional.pad(sample, (0, case["docs"] * hi - sample.numel()), value=-1)
    tokens = torch.nn.functional.pad(tokens, (0, case["encode_docs"] * hi - tokens.numel()), value=-1)
    return {"merges": merges, "sample": sample, "sample_offsets": sample_off, "rows": rows, "tokens": tokens, "offsets": off}


# ------------------------------------------------------------------------------------------------------------ work
def _mean_ctx(case):
    return case["ctx"] * (0.75 if case["ragged"] else 1.0)


def _forward(s, rows, ctx, seqs, lm_head):
    """Bytes and operations of one pass of `rows` rows in all over `seqs` sequences of `ctx` committed tokens: every
    weight once, the cached K and V once, the new ones written; two operations per weight and row, and the attention."""
    esz = 4 if s.dtype == "f32" else 2
    params = s.matmul_params() - (0 if lm_head else s.vocab * s.d_model)
    kv = s.kv_bytes_per_token()
    return (params * esz + rows * s.d_model * esz + seqs * ctx * kv + rows * kv,
            2.0 * params * rows + 4.0 * s.n_layers * s.q_dim * rows * ctx)


def work(case):
    kind = case["kind"]
    if kind in ("task", "tokenizer"):
        cfg = configs.get(case["recipe"])
        mean = (cfg.corpus.len_lo + cfg.corpus.len_hi) / 2
        if kind == "task":                       # the corpus once for the statistics and once for the tables
            return {"bytes": 2.0 * case["docs"] * (mean * 4 + 8), "flops": 0.0}
        rows = case["budget"] * cfg.model.d_model * 2.0
        return {"bytes": 2.0 * (case["docs"] + case["encode_docs"]) * (mean * 4 + 8) + rows * (1 + case["n_max"]), "flops": 0.0}
    s, _ = _shape(case["model"])
    B, ctx = case["batch"], _mean_ctx(case)
    if kind == "step":
        nbytes, flops = _forward(s, B * (case["k"] + 1), ctx, B, True)
        return {"bytes": nbytes + 4.0 * B * ctx, "flops": flops}       # the drafter reads the committed tokens
    nbytes, flops = _forward(s, B * (ctx - 1), ctx / 2, 0, False)      # a prompt attends to itself
    if kind == "generate":
        # every draft accepted is the least number of steps
        steps = -(-case["new"] // (case["k"] + 1))
        per = _forward(s, B * (case["k"] + 1), ctx + case["new"] / 2, B, True)
        nbytes, flops = nbytes + steps * per[0], flops + steps * per[1]
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    kind = case["kind"]
    if kind == "task":
        return {"rel": 1e-9}                     # counts and drafts exact; entropies are double-precision sums
    if kind == "tokenizer":
        return "exact"
    if case["model"] == "tiny-f32":
        return {"rel": 1e-5, "max": 1e-3}
    # bf16 cache: an element on the other side of a rounding boundary moves by 2^-8 of its value, and later layers see it;
    # token rows may differ at ties of the two largest logits
    return {"rel": 1e-2, "max": 0.2, "differ": 0.01}
