"""First steps of up to four sequences as a chain of launches (three bf16 terms an activation): one to four rows, rows and columns that
leave the last weight tile ragged, k ranges of one k block and of more than eight, beside the prefill and behind it.  Against the oracle, and
the step alone, on the GPU's own cache: a quarter of what dropping the third term moves the oracle bounds its error (sums of up to eight k
blocks go through few instructions that round towards zero, and partial sums are added in fp32)."""
import pytest

import workloads as wl
from parity_util import TOL, assert_first_tokens, compare_prefill, make_session, rel_fro
from recorded_graph import recorded_prefill
from test_step_mma_gpu import _step, _two_terms

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,heads,d,ffn,lens", [
    (64, (24, 8), 1544, 2568, [9, 130, 64]),               # 1544 = 12 x 128 + 8 rows, 24 x 64 + 8 k
    (128, (12, 3), 1544, 2568, [1, 65, 200, 33]),
    (64, (40, 8), 2056, 2056, [1500, 1400, 1300]),         # more than 4096 tokens: the step follows the prefill
], ids=str)
def test_first_step_as_a_chain_matches_oracle(hd, heads, d, ffn, lens):
    pair = wl.PairCfg("chain3", wl.uniform_model(2, 128, 2, 1, 64, 128, 300), wl.uniform_model(2, d, heads[0], heads[1], hd, ffn, 300), (0, 1))
    W = wl.make_weights(pair, seed=9, regime="fanin")
    g = recorded_prefill(pair, lens, W)
    assert g.find("step_gemm_kernel") and not g.find("step_mega")
    pr = wl.custom_prompts(300, lens, seed=9)
    s = make_session(pair, W, pr)
    try:
        ek, ev, el, tally = compare_prefill(s, pair, W, pr)
        assert_first_tokens(tally, TOL[pair.dtype], "chain3")
        logits = s.logits.cpu().numpy()
        for b, n in enumerate(lens):
            cache = [s.cache.gather(i, b, n) for i in range(2)]
            token = int(pr.seq(b)[-1])
            want = _step(pair, W, token, cache)[0]
            err, two = rel_fro(logits[b], want), rel_fro(_step(pair, W, token, cache, _two_terms)[0], want)
            print(f"sequence {b}: {err:.2e}, two terms {two:.2e}")
            assert err <= 0.25 * two
    finally:
        s.close()
