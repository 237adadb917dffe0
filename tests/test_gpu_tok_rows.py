"""Rows of added tokens, in order, by warps that wait for one another: chains in which every added token needs the one before, more added tokens than a chunk holds, widths
beside those of a block's columns, tokens that need rows of an earlier chunk and of their own.  Bit-exact against the oracle."""
import numpy as np
import pytest
import torch

from oracle import tasc_tok as T
from tests.gpu_harness import need_gpu
from workload.weights import round_to_bf16


def make_merges(kind, n, vocab, r):
    out = []
    for i in range(n):
        if kind == "chain":                                    # each added token needs the one before it
            g = [vocab + i - 1 if i else 1, 2]
        elif kind == "flat":                                   # none needs another
            g = r.integers(0, vocab, r.integers(2, 7)).tolist()
        else:                                                  # any token that exists, the newest ones often
            g = [int(max(0, vocab + i - 1 - r.geometric(0.05))) if r.random() < 0.5 else int(r.integers(0, vocab + i)) for _ in range(r.integers(2, 7))]
        out.append(tuple(g))
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("kind,n", [("flat", 1), ("chain", 70), ("mixed", 256), ("mixed", 257), ("flat", 2100), ("chain", 1100), ("mixed", 3000)])
@pytest.mark.parametrize("d", [1, 31, 32, 33, 96])
def test_rows_in_order(kind, n, d):
    b = need_gpu()
    r = np.random.default_rng(n + d)
    vocab = 50
    merges = make_merges(kind, n, vocab, r)
    m = np.full((n, 6), -1, np.int32)
    for i, g in enumerate(merges):
        m[i, :len(g)] = g
    md = torch.from_numpy(m).cuda()
    E = r.standard_normal((vocab, d)).astype(np.float32)
    assert np.array_equal(b.tasc_tok_init_rows(torch.from_numpy(E).cuda(), md).cpu().numpy(), T.new_rows(E, merges, vocab, bf16=False))
    E16 = round_to_bf16(E)
    got = b.tasc_tok_init_rows(torch.from_numpy(E16).cuda().bfloat16(), md).float().cpu().numpy()
    assert np.array_equal(got, T.new_rows(E16, merges, vocab, bf16=True))


@pytest.mark.gpu
@pytest.mark.parametrize("at", [0, 5, 255, 256, 1500])
@pytest.mark.parametrize("bad", [(60 + 1500, 1), (60, -1)])
def test_a_row_that_cannot_be_made_is_refused(at, bad):
    """A constituent that does not exist yet, and an added token of one constituent, in any chunk."""
    b = need_gpu()
    r = np.random.default_rng(at)
    n, vocab = 1501, 60
    m = np.full((n, 6), -1, np.int32)
    m[:, :2] = r.integers(0, vocab, (n, 2))
    m[at, :2] = bad
    with pytest.raises(b.TascError):
        b.tasc_tok_init_rows(torch.zeros((vocab, 40), device="cuda"), torch.from_numpy(m).cuda())
