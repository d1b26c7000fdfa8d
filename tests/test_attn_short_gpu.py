"""Prompt attention of short sequences: lengths at the edges of its 64-query and 64-key tiles and of a warp's 16 rows, both head widths,
bfloat16 (prefill) and IEEE-half operands with a remainder (training-time forward), against the oracle.  The rule that picks the form
of a call is looked at on the sizes themselves: these calls take the short form."""
import pytest

import workloads as wl
from oracle import kvp_oracle as orc
from parity_util import TOL, assert_first_tokens, compare_prefill, make_session, rel_fro

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,heads,lens", [(64, (4, 1), [1]), (64, (4, 2), [16, 17, 63, 64, 65, 1, 15]), (64, (20, 5), [128, 127, 129, 64, 192, 31, 33, 2]),
                                           (128, (3, 1), [1, 63, 64, 65]), (128, (4, 4), [128, 16, 100, 127, 5])], ids=str)
def test_short_prompts_match_oracle(hd, heads, lens):
    aux = wl.uniform_model(3, 192, heads[0], heads[1], hd, 192, 300)
    pair = wl.PairCfg("short", aux, wl.uniform_model(3, 128, 2, 1, hd, 128, 300), (0, 1, 2))
    W = wl.make_weights(pair, seed=8, regime="fanin")
    pr = wl.custom_prompts(300, lens, seed=8)
    s = make_session(pair, W, pr)
    try:
        ek, ev, el, tally = compare_prefill(s, pair, W, pr)
        print(f"K {ek:.2e} V {ev:.2e} logits {el:.2e}")
        assert_first_tokens(tally, TOL[pair.dtype], "short")
    finally:
        s.close()


@pytest.mark.parametrize("hd,lens", [(64, [65, 1, 64, 100, 16]), (128, [64, 65, 3])], ids=str)
def test_training_forward_of_short_prompts_matches_oracle(hd, lens):
    import torch
    pair = wl.PairCfg("short", wl.uniform_model(2, 128, 2, 1, hd, 128, 300), wl.uniform_model(3, 192, 4, 2, hd, 192, 300), (0, 1, 1))
    W = wl.make_weights(pair, seed=8, regime="fanin")
    pr = wl.custom_prompts(300, lens, seed=8)
    s = make_session(pair, W, pr)
    try:
        toks = torch.from_numpy(pr.tokens).to(s.device)
        s.prefill_predict(toks, lens)
        logits, l1_k, l1_v = s.train_forward(toks, lens)
        s.poll()
        logits, t0 = logits.cpu().numpy(), 0
        for b in range(pr.batch):
            want = orc.train_forward(pair, W, pr.seq(b))[0]
            assert max(rel_fro(logits[t0 + t], want[t]) for t in range(lens[b])) <= TOL["bf16"]
            t0 += lens[b]
    finally:
        s.close()
