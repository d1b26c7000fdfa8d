"""Kernels that give a row of the model width, of the vocabulary or of a layer's keys to a few threads: widths at which their
16-byte pieces, their pieces per thread and their scalar forms begin and end, against the oracle."""
import numpy as np
import pytest

import workloads as wl
from oracle import kvp_oracle as orc
from parity_util import TOL, make_session, rel_fro

pytestmark = pytest.mark.gpu


# d_model: 512 is the last width of one warp a row, 2048 the last of 4 pieces a thread, 4096 the last that is held in registers;
# 66, 70: no whole 16-byte pieces.  vocab: no whole pieces, one more than a trip of the block's four loads.
@pytest.mark.parametrize("dtype,d,vocab", [("bf16", 512, 97), ("bf16", 516, 16388), ("bf16", 2056, 640), ("bf16", 4100, 333), ("f32", 66, 101),
                                           ("f32", 4096, 64), ("bf16", 70, 4097)], ids=str)
def test_row_widths_match_oracle(dtype, d, vocab):
    import torch
    pair = wl.PairCfg("rows", wl.uniform_model(2, d, 2, 1, 64, 128, vocab), wl.uniform_model(2, d, 2, 1, 64, 128, vocab), (0, 1), dtype=dtype)
    W = wl.make_weights(pair, seed=4, regime="fanin")
    lens = [9, 1, 64, 30, 66]
    pr = wl.custom_prompts(vocab, lens, seed=4)
    s = make_session(pair, W, pr, extra_len=1)
    tol = TOL[dtype]
    try:
        logits, first = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        logits, first = logits.cpu().numpy(), first.cpu().numpy()
        ref = orc.prefill_predict(pair, W, pr)
        caches = {b: ref[b][0] for b in range(pr.batch)}
        for b in range(pr.batch):
            assert rel_fro(logits[b], ref[b][1]) <= tol
            assert int(first[b]) == int(np.argmax(logits[b]))
        nxt = np.arange(pr.batch, dtype=np.int32) % vocab
        logits, tok = s.decode_step(torch.from_numpy(nxt).to(s.device), lens)
        s.poll()
        logits = logits.cpu().numpy()
        for b in range(pr.batch):
            want, _ = orc.decode_step(pair, W, int(nxt[b]), caches[b])
            assert rel_fro(logits[b], want) <= tol
            assert int(tok[b]) == int(np.argmax(logits[b]))
    finally:
        s.close()


def _first_tokens(pair, W, pr):
    import torch
    s = make_session(pair, W, pr)
    try:
        logits, first = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), [int(n) for n in pr.lengths])
        s.poll()
        return logits.cpu().numpy(), first.cpu().tolist()
    finally:
        s.close()


# 16390: element by element; 16388, 32000: 16-byte pieces, four a thread and trip of 16384 elements
@pytest.mark.parametrize("vocab,tied", [(16390, range(16390)), (16388, range(16388)), (32000, range(32000)),
                                        (32000, [4 * 40 + 16384, 4 * 40]),             # one thread, on two trips
                                        (32000, [4 * 7 + 4096, 4 * 7 + 8192 + 3]),     # one thread, two of a trip's four pieces
                                        (32000, [4 * 9 + 1, 4 * 9 + 2]),               # one piece
                                        (32000, [4 * 33, 4 * 34 + 3]),                 # neighbouring lanes
                                        (32000, [4 * 1023 + 3, 4 * 31 + 16384]),       # two warps, the lower index in the later one
                                        (32000, [31999, 16000, 20000]), (16388, [16387, 16384]), (16390, [16389, 5001])],
                         ids=lambda v: str(v)[:30].replace(" ", ""))
def test_argmax_takes_the_lowest_index_of_a_tie(vocab, tied):
    """Rows of the head that are the same give logits that are the same (one k block: d_model 64)."""
    pair = wl.PairCfg("tie", wl.uniform_model(1, 64, 1, 1, 64, 64, vocab), wl.uniform_model(1, 64, 1, 1, 64, 64, vocab), (0,))
    W = wl.make_weights(pair, seed=4)
    pr = wl.custom_prompts(vocab, [5] * 5, seed=4)
    pr.tokens[:] = np.tile(pr.tokens[:5], 5)
    head = W["base.lm_head"].copy()
    if len(tied) < vocab:        # four times the row whose logit is the largest, and so far above all others
        head[list(tied)] = 4 * head[_first_tokens(pair, W, pr)[1][0]]
    else:
        head[:] = 0
    W["base.lm_head"] = head
    logits, first = _first_tokens(pair, W, pr)
    assert first == [min(tied)] * 5
    for row in logits:
        assert sorted(np.flatnonzero(row == row.max())) == sorted(tied)
