"""Captured steps whose draft or verify step follows what is not a kernel of the library: a copy, a memset, another stream's event.  The first
kernels of both may be set up while the kernel before them runs; in a graph they have to wait for nodes that are no kernels too."""
import numpy as np
import pytest
import torch

from tests.gpu_harness import make_setup, need_gpu
from workload import configs


@pytest.mark.gpu
@pytest.mark.parametrize("before", ["copy", "memset", "event"])
@pytest.mark.parametrize("index,B", [(0, 1), (1, 1), (1, 5)])        # float32 in a cluster, one-kernel layers, five kernels per layer
def test_replayed_steps_wait_for_what_comes_before_them(index, B, before):
    b = need_gpu()
    cfg = configs.shrunk(configs.get(index), n_layers=2, vocab=512, n_docs=300)
    s = make_setup(cfg, oracle_ngrams=False)
    k, P = 4, 40
    rng = np.random.default_rng(B)
    texts = [torch.from_numpy(rng.integers(0, 512, (B, P + 2 * (k + 1))).astype(np.int32)).cuda() for _ in range(2)]
    other = [torch.from_numpy(rng.integers(0, 512, (B, k)).astype(np.int32)).cuda() for _ in range(2)]
    src, src_drafts, length0 = texts[0].clone(), other[0].clone(), torch.full((B,), P, dtype=torch.int32, device="cuda")
    tokens, length = texts[0].clone(), length0.clone()
    drafts = torch.zeros((B, k), dtype=torch.int32, device="cuda")
    pool, bt, kv = s.model.new_kv(B, tokens.shape[1] + b.MAX_ROWS)
    ws = s.model.new_workspace(B, k)
    seqs = b.make_seqs(tokens, length)
    b.tasc_prefill(s.model, kv, seqs, B, P, ws)
    side = torch.cuda.Stream()

    def step():
        main = torch.cuda.current_stream()
        if before == "event":
            side.wait_stream(main)
            with torch.cuda.stream(side):
                torch.cuda._sleep(200000)
                torch.add(src, 0, out=tokens)
                length.copy_(length0)
            main.wait_stream(side)
        else:
            tokens.copy_(src)
            length.copy_(length0)
        b.tasc_draft(s.drafter, tokens, length, k, out=drafts)
        kept = drafts.clone()
        if before == "memset":
            drafts.zero_()
        elif before == "copy":
            drafts.copy_(src_drafts)
        else:
            side.wait_stream(main)
            with torch.cuda.stream(side):
                torch.cuda._sleep(200000)
                torch.add(src_drafts, 0, out=drafts)
            main.wait_stream(side)
        acc, nxt, tgt, logits = b.tasc_verify_step(s.model, kv, seqs, drafts, ws, want_targets=True, want_logits=True)
        return kept, acc, nxt, tgt, logits, tokens, length

    want = []
    for i in range(2):
        src.copy_(texts[i])
        src_drafts.copy_(other[i])
        want.append([t.clone() for t in step()])
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=stream):
        got = step()
    for i in (0, 1, 1, 0):
        src.copy_(texts[i])
        src_drafts.copy_(other[i])
        graph.replay()
        for g, w in zip(got, want[i]):
            assert torch.equal(g, w)
    b.tasc_poll_status(ws)
