"""The enrichment's look-ups of changed windows, which all threads of a CTA share: documents with more changed windows than a warp's list
holds, more documents than a CTA has warps, documents at the lengths where another way of rewriting them begins.  Bit-exact."""
import numpy as np
import pytest

from tests.gpu_harness import need_gpu
from tests.test_gpu_tasc_tok import check_enrich, flat


@pytest.mark.gpu
@pytest.mark.parametrize("n_max", [2, 4, 6])
@pytest.mark.parametrize("length,n_docs", [(3, 20), (58, 900), (130, 40), (255, 33), (256, 300), (257, 33)])
def test_documents_full_of_occurrences(length, n_docs, n_max):
    """Every second pair of a document is the n-gram of the first rounds: hundreds of windows per document change at once.  Some documents
    without it among them."""
    b = need_gpu()
    r = np.random.default_rng(length + n_max)
    docs = []
    for i in range(n_docs):
        d = np.where(r.random(length) < 0.2, r.integers(4, 40, length), np.tile([1, 2], length)[:length])
        docs.append((r.integers(4, 40, length) if i % 7 == 3 else d).tolist())
    check_enrich(b, *flat(docs), 40, 12, n_max)


@pytest.mark.gpu
@pytest.mark.parametrize("every", [2, 9, 60])
@pytest.mark.parametrize("n_docs", [40, 1500])
def test_long_documents_among_short_ones(n_docs, every):
    """A CTA with a document of more than 256 tokens hands its documents out one by one, the others a document per warp at a time: both in
    a round, documents that are long in the first rounds and short in later ones."""
    b = need_gpu()
    r = np.random.default_rng(n_docs + every)
    docs = []
    for i in range(n_docs):
        length = int(r.integers(257, 700) if i % every == 0 else r.integers(0, 120))
        docs.append(np.where(r.random(length) < 0.3, r.integers(4, 40, length), np.tile([1, 2, 3], length // 3 + 1)[:length]).tolist())
    check_enrich(b, *flat(docs), 40, 12, 4)
