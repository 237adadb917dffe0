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
