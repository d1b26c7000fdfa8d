"""Prompt attention of short sequences: lengths at the edges of its 64-query and 64-key tiles and of a warp's 16 rows, both head widths,
bfloat16 (prefill) and IEEE-half operands with a remainder (training-time forward), against the oracle.  The recorded graph says that
these calls take the short form, and that each of the three forms is taken by the calls it was measured to be the fastest for."""
import pytest

import workloads as wl
from oracle import kvp_oracle as orc
from parity_util import TOL, assert_first_tokens, compare_prefill, make_session, rel_fro
from recorded_graph import Recorded, recorded_prefill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,heads,lens", [(64, (4, 1), [1]), (64, (4, 2), [16, 17, 63, 64, 65, 1, 15]), (64, (20, 5), [128, 127, 129, 64, 192, 31, 33, 2]),
                                           (128, (3, 1), [1, 63, 64, 65]), (128, (4, 4), [128, 16, 100, 127, 5])], ids=str)
def test_short_prompts_match_oracle(hd, heads, lens):
    aux = wl.uniform_model(3, 192, heads[0], heads[1], hd, 192, 300)
    pair = wl.PairCfg("short", aux, wl.uniform_model(3, 128, 2, 1, hd, 128, 300), (0, 1, 2))
    W = wl.make_weights(pair, seed=8, regime="fanin")
    pr = wl.custom_prompts(300, lens, seed=8)
    g = recorded_prefill(pair, lens, W)
    assert len(g.find("attn_mma_kernelILi%dELb0E" % hd)) == 2 and not g.find("attn_tc_kernel")
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

    import paper_2410_08391_b200 as kvp
    pair = wl.PairCfg("short", wl.uniform_model(2, 128, 2, 1, hd, 128, 300), wl.uniform_model(3, 192, 4, 2, hd, 192, 300), (0, 1, 1))
    W = wl.make_weights(pair, seed=8, regime="fanin")
    pr = wl.custom_prompts(300, lens, seed=8)
    s = make_session(pair, W, pr)
    try:
        toks = torch.from_numpy(pr.tokens).to(s.device)
        s.prefill_predict(toks, lens)
        logits, l1_k, l1_v = s.train_forward(toks, lens)
        s.poll()
        g = Recorded(s, lambda: kvp.kvp_train_forward(s.h, toks, lens, s.cache, s.train_ws, logits, l1_k, l1_v, s.stream))
        assert len(g.find("attn_mma_kernelILi%dELb1E" % hd)) == 2 * 3 - 1 and not g.find("attn_tc_kernel")
        s.poll()
        logits, t0 = logits.cpu().numpy(), 0
        for b in range(pr.batch):
            want = orc.train_forward(pair, W, pr.seq(b))[0]
            assert max(rel_fro(logits[t0 + t], want[t]) for t in range(lens[b])) <= TOL["bf16"]
            t0 += lens[b]
    finally:
        s.close()


@pytest.mark.parametrize("heads,hd,lens,form", [((20, 5), 64, [59] * 64, 0), ((20, 5), 64, [59], 0), ((20, 5), 64, [1024], 1), ((20, 5), 64, [700], 1),
                                                ((12, 3), 128, [4096], 2), ((12, 3), 128, [3500, 1200, 2000], 2)], ids=str)
def test_form_of_the_prompt_attention(heads, hd, lens, form):
    """0: this file's kernel; 1, 2: the tcgen05 kernel with that many 128-query tiles a CTA (its grid: query heads x such pieces of the prompts)."""
    aux = wl.uniform_model(2, heads[0] * hd, heads[0], heads[1], hd, 128, 300)
    pair = wl.PairCfg("form", aux, wl.uniform_model(2, 128, 2, 1, hd, 128, 300), (0, 1))
    g = recorded_prefill(pair, lens)
    short, tc = g.find("attn_mma_kernelILi%dELb0E" % hd), g.grids("attn_tc_kernel")
    if form == 0:
        assert len(short) == 1 and not tc
    else:
        items = sum((n + 128 * form - 1) // (128 * form) for n in lens)
        assert not short and len(tc) == 1 and items in tc[0] and heads[0] in tc[0]
