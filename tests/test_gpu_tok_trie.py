"""The added tokens' trie that encoding walks: few edges and many, as its table grows; expansions that begin with one another, or are the same;
none at all.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import tasc_tok as T
from tests.gpu_harness import need_gpu
from tests.test_gpu_tasc_tok import flat, to_dev


@pytest.mark.gpu
@pytest.mark.parametrize("n,vocab", [(0, 9), (1, 9), (60, 3), (85, 4000), (102, 60000), (103, 60000), (1500, 50), (2000, 30000)])
def test_encoding_with_any_number_of_edges(n, vocab):
    b = need_gpu()
    r = np.random.default_rng(n + vocab)
    merges = []
    for i in range(n):                                          # base tokens and added ones: the newest ones begin with older ones' expansions
        while True:
            g = tuple(int(t) for t in r.integers(0, vocab + (i if r.random() < 0.3 else 0), r.integers(2, 7)))
            if len(T.expansion(merges + [g], vocab, vocab + i)) <= 40:
                break
        merges.append(g)
    m = np.full((n, 6), -1, np.int32)
    for i, g in enumerate(merges):
        m[i, :len(g)] = g
    docs = []
    for _ in range(50):                                         # expansions, whole and cut short, between other tokens
        d = []
        for _ in range(int(r.integers(0, 12))):
            e = T.expansion(merges, vocab, vocab + int(r.integers(0, n))) if n else [1, 2]
            d += list(e[:int(r.integers(1, len(e) + 1))] if r.random() < 0.3 else e) + r.integers(0, vocab, int(r.integers(0, 3))).tolist()
        docs.append([int(t) for t in d])
    toks, offs = b.tasc_tok_encode(*to_dev(*flat(docs)), vocab, torch.from_numpy(m).cuda())
    wt, wo = flat([T.encode(d, merges, vocab) for d in docs])
    assert np.array_equal(offs.cpu().numpy(), wo) and np.array_equal(toks.cpu().numpy(), wt)
