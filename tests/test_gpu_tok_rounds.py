"""The merge rounds of the tokenizer enrichment where they leave their usual way: more n-grams near the best than the list of
candidates holds, ties of more n-grams than are looked for by their tokens, more documents with the n-gram than a CTA lists at once,
documents too long for shared memory.  Bit-exact against the oracle, like tests/test_gpu_tasc_tok.py."""
import numpy as np
import pytest

from tests.gpu_harness import need_gpu
from tests.test_gpu_tasc_tok import check_enrich, flat


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
