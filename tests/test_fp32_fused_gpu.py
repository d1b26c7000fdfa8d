"""fp32 mode's products with the norm in front, the rotation and SwiGLU behind them, at the edges of 32 x 32 and 64 x 64 tiles and of
their 64 and 32 k at a time, against the oracle (sums of some hundred fp32 products in another order: 1e-4)."""
import pytest

import workloads as wl
from parity_util import TOL, assert_first_tokens, compare_prefill, make_session
from recorded_graph import recorded_prefill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,heads,hd,ffn,lens,tile", [
    (8, (1, 1), 2, 8, [1], 32),                                    # smaller than a tile everywhere
    (64, (4, 4), 16, 172, [64], 32),                               # ffn no multiple of 64: gate and up rows in blocks of unequal size
    (100, (3, 1), 34, 71, [33, 31], 32),                           # halves of 17 columns straddle tiles; k and columns ragged
    (68, (6, 3), 128, 128, [65], 32),                              # a head is four tiles wide
    (132, (8, 2), 62, 450, [700, 200, 173], 64),                   # 1073 rows: 64 x 64 tiles, all ragged
], ids=str)
def test_fp32_products_match_oracle(d, heads, hd, ffn, lens, tile):
    pair = wl.PairCfg("fp32", wl.uniform_model(2, d, heads[0], heads[1], hd, ffn, 97), wl.uniform_model(2, 32, 2, 1, 8, 40, 97), (0, 1), dtype="f32")
    W = wl.make_weights(pair, seed=4, regime="fanin")
    g = recorded_prefill(pair, lens, W)
    assert g.find("gemm_rope_split_kernelILi%dE" % tile) and not g.find("rmsnorm|swiglu_kernel")
    pr = wl.custom_prompts(97, lens, seed=4)
    s = make_session(pair, W, pr)
    try:
        ek, ev, el, tally = compare_prefill(s, pair, W, pr)
        print(f"K {ek:.2e} V {ev:.2e} logits {el:.2e}")
        assert_first_tokens(tally, TOL[pair.dtype], "fp32")
    finally:
        s.close()
