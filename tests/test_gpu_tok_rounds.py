"""The merge rounds of the tokenizer enrichment where they leave their usual way: more n-grams near the best than the list of
candidates holds, ties of more n-grams than are looked for by their tokens, more documents with the n-gram than a CTA lists at once,
documents too long for shared memory.  Bit-exact against the oracle, like tests/test_gpu_tasc_tok.py."""
import numpy as np
import pytest
import torch

from tests.gpu_harness import need_gpu
from tests.test_gpu_tasc_tok import check_enrich, flat, merges_as_tuples, to_dev


@pytest.mark.gpu
@pytest.mark.parametrize("n_docs,repeats,budget", [(700, 2, 6), (1500, 1, 5), (4, 3, 12)])
def test_more_equal_ngrams_than_the_list_holds(n_docs, repeats, budget):
    """Documents of three tokens that occur nowhere else, each `repeats` times: every pair and triple has the same count, so that
    thousands tie, then a few dozen; one frequent phrase first."""
    b = need_gpu()
    docs = [[3 * i + 20, 3 * i + 21, 3 * i + 22] for i in range(n_docs)] * repeats + [[1, 2, 3, 4]] * 9
    check_enrich(b, *flat(docs), 3 * n_docs + 30, budget, 3)


@pytest.mark.gpu
@pytest.mark.parametrize("n_docs,tail", [(152000, 0), (160000, 300)])
def test_more_documents_than_a_cta_lists(n_docs, tail):
    """All documents hold the first n-grams: over 1,024 of them start in each CTA's share (148 CTAs).  Two long ones among them."""
    b = need_gpu()
    r = np.random.default_rng(n_docs)
    docs = [[5, 6] if i % 3 else [5, 6, 7] for i in range(n_docs)]
    if tail:
        docs[1000] = r.integers(5, 9, tail).tolist()
        docs[90000] = r.integers(5, 9, 1000).tolist()
    check_enrich(b, *flat(docs), 16, 3, 3)


@pytest.mark.gpu
@pytest.mark.parametrize("n_max", [2, 4, 6])
def test_candidates_come_and_go(n_max):
    """Phrases with slowly falling counts that share tokens: the list is made anew several times, n-grams with the new tokens rise past
    its floor, others fall below it."""
    b = need_gpu()
    r = np.random.default_rng(n_max)
    phrases = [r.integers(0, 30, r.integers(2, 7)).tolist() for _ in range(60)]
    docs = [sum((phrases[min(59, int(r.zipf(1.3)))] for _ in range(r.integers(1, 12))), []) for _ in range(1500)]
    check_enrich(b, *flat(docs), 30, 80, n_max)


# (the hash of csrc/ngram_table.cuh: key_make(2), key_put, key_hash)
def first_pair(x, y, cap):
    """First pair of slots that the table of `cap` slots looks at for the bigrams (x[i], y[i])."""
    x, y = x.astype(np.uint64), y.astype(np.uint64)
    u = np.uint64
    with np.errstate(over="ignore"):
        h = (x | y << u(20)) * u(0x9E3779B97F4A7C15) ^ u(((1 << 63 | 2 << 56) + 0xD6E8FEB86659FD93) % (1 << 64))
        h = (h ^ h >> u(32)) * u(0xD6E8FEB86659FD93)
        h = (h ^ h >> u(29)) * u(0x9E3779B97F4A7C15)
    return (h ^ h >> u(32)) & u(cap // 2 - 1)


@pytest.mark.gpu
@pytest.mark.parametrize("early", [1022, 1023, 1024, 1025])
def test_a_list_that_is_just_full(early):
    """The list of candidates holds 1,024.  All candidates lie in chunks of the table that one warp looks through in turn: `early` with
    the same count, the last of them alone in its chunk, then the next-best n-gram, then the best.  Where the early ones are exactly
    1,024, the two behind them have to be seen to be missing."""
    b = need_gpu()
    r = np.random.default_rng(17)
    vocab, cap, chunk, warp = 2 ** 20 - 8, 2 ** 24, 128, 777
    warps = 32 * torch.cuda.get_device_properties(0).multi_processor_count
    assert cap // chunk > 26 * warps + warp
    # over four million windows of other n-grams, so that the table has 2^24 slots
    filler = r.integers(0, vocab, (66, 1000), dtype=np.int64)
    x, y = r.integers(0, vocab, (2, 16_000_000), dtype=np.int64)
    pair = first_pair(x, y, cap)
    turn, whose = np.divmod(pair // np.uint64(chunk // 2), np.uint64(warps))     # a chunk's place among its warp's, and the warp
    # n-grams by chunk, one to a pair of slots that no other n-gram looks at first: all lie there
    used = set(first_pair(filler[:, :-1].ravel(), filler[:, 1:].ravel(), cap).tolist())
    chunks = [[] for _ in range(27)]
    for i in np.flatnonzero((whose == warp) & (turn < 27)):
        if int(pair[i]) not in used:
            used.add(int(pair[i]))
            chunks[int(turn[i])].append((int(x[i]), int(y[i])))
    chosen = sum(chunks[:24], [])[:early - 1] + chunks[24][:1]
    assert len(chosen) == early
    next_best, best = chunks[25][0], chunks[26][0]
    counts = [(best, 200), (next_best, 180)] + [(g, 160) for g in chosen]
    docs = np.concatenate([np.tile(np.array(g, np.int32), n) for g, n in counts] + [np.tile(filler.astype(np.int32).ravel(), 67)])
    lens = np.concatenate([np.full(sum(n for _, n in counts), 2), np.full(66 * 67, 1000)])
    assert cap // 4 < (lens - 1).sum() <= cap // 2
    merges, _, _ = b.tasc_tok_enrich(*to_dev(docs, np.concatenate([[0], np.cumsum(lens)])), vocab, 4, 2)
    assert merges_as_tuples(merges) == [best, next_best, chosen[0], chosen[1]]
