"""The scan of the corpus (how many tokens follow in the document, token counts) where documents meet the edges of its runs of 4,096
positions and of the 255 tokens it tells apart: tables and statistics against the oracles."""
import numpy as np
import pytest

from tests.gpu_harness import need_gpu
from tests.test_gpu_corpus_stats import both
from tests.test_gpu_drafter import assert_tables_equal, build_both


def documents(kind, r):
    if kind == "one":
        return [9000]                                            # a document longer than two runs
    if kind == "edges":
        return [4096, 4095, 1, 4097, 255, 256, 257, 258, 0, 4096]
    if kind == "empty":
        return [0] * 700 + [3] + [0] * 5000 + [4093] + [0] * 3 + [2, 0]
    return r.integers(0, 600, 400).tolist()


@pytest.mark.gpu
@pytest.mark.parametrize("kind", ["one", "edges", "empty", "mixed"])
def test_documents_at_the_edges_of_a_run(kind):
    need_gpu()
    r = np.random.default_rng(7)
    lens = np.array(documents(kind, r))
    vocab = 50
    offsets = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    tokens = r.integers(0, vocab, offsets[-1]).astype(np.int32)
    both(tokens, offsets, vocab)
    _, drafter, ngrams = build_both(tokens, offsets, 3, 2, vocab)
    assert_tables_equal(drafter, ngrams)
