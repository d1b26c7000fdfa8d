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


def test_argmax_takes_the_lowest_index_of_a_tie():
    """Zero weights in front of the head: every logit is the same, in every row."""
    import torch
    pair = wl.PairCfg("tie", wl.uniform_model(1, 64, 1, 1, 64, 64, 16390), wl.uniform_model(1, 64, 1, 1, 64, 64, 16390), (0,))
    W = wl.make_weights(pair, seed=4)
    W["base.lm_head"] = np.zeros_like(W["base.lm_head"])
    lens = [3, 4, 5, 6, 7]
    pr = wl.custom_prompts(16390, lens, seed=4)
    s = make_session(pair, W, pr)
    try:
        logits, first = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        assert first.cpu().tolist() == [0] * 5 and float(logits.abs().max()) == 0.0
    finally:
        s.close()
