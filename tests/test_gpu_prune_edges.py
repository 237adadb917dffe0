"""Order n + 1 is counted from the frequent windows of order n, four positions per thread and a bit per slot of the table: corpora that
end at and beside the edges of a thread's, a warp's and a block's positions, against the oracle's tables."""
import numpy as np
import pytest

from tests.test_gpu_drafter import assert_tables_equal, build_both


@pytest.mark.gpu
@pytest.mark.parametrize("n_tokens", [3, 4, 5, 127, 128, 129, 1023, 1024, 1025, 4099])
def test_corpora_that_end_at_an_edge(n_tokens):
    r = np.random.default_rng(n_tokens)
    tokens = (r.random(n_tokens) ** 2 * 7).astype(np.int32)
    for offsets in ([0, n_tokens], [0, n_tokens // 3, n_tokens - 1, n_tokens]):
        _, drafter, ngrams = build_both(tokens, np.array(offsets, dtype=np.int64), 4, 2, 7)
        assert_tables_equal(drafter, ngrams)
