"""The tensor-core GEMM at every tile width and both ways of cutting the work: rows, columns and k that leave the last tile, the last
piece of a cache row and the last k block ragged, against the oracle.  Which width a size takes is the launcher's rule (76 SMs beside
a step of up to four sequences, 148 otherwise); the sizes are some that it cuts that way."""
import pytest

import workloads as wl
from parity_util import TOL, assert_first_tokens, compare_prefill, make_session
from recorded_graph import recorded_prefill

pytestmark = pytest.mark.gpu
TWO = [1000, 999]                # 1999 rows = 15.6 row blocks


@pytest.mark.parametrize("d,ffn,heads,base_kv,lens", [
    (72, 128, (1, 1), 1, [70]),             # 128 columns, one ragged tile
    (520, 200, (3, 1), 2, TWO),             # residual 160: 3.25 tiles
    (648, 136, (7, 1), 9, TWO),             # residual 192: 3.4 tiles; q / k / v 576 = 3 x 192; predictor 576
    (776, 72, (3, 3), 3, TWO),              # residual 224: 3.5 tiles
    (904, 64, (2, 1), 1, TWO),              # residual 256: 3.5 tiles
    (264, 4104, (2, 2), 2, [70, 3]),        # shares of the k blocks: 65 k blocks of three 128-wide tiles
    (1032, 2056, (4, 1), 9, [301, 200, 190, 64, 35, 1000]),     # 148 SMs, shares of 256-wide tiles
], ids=str)
def test_every_cut_matches_oracle(d, ffn, heads, base_kv, lens):
    aux = wl.uniform_model(2, d, heads[0], heads[1], 64, ffn, 500)
    pair = wl.PairCfg("cuts", aux, wl.uniform_model(2, 128, base_kv, base_kv, 64, 128, 500), (0, 1))
    W = wl.make_weights(pair, seed=6, regime="fanin")
    pr = wl.custom_prompts(500, lens, seed=6)
    s = make_session(pair, W, pr)
    try:
        ek, ev, el, tally = compare_prefill(s, pair, W, pr)
        print(f"K {ek:.2e} V {ev:.2e} logits {el:.2e}")
        assert_first_tokens(tally, TOL[pair.dtype], "cuts")
    finally:
        s.close()


def test_folded_norm_with_ragged_columns_matches_oracle():
    """Enough tokens for the residual GEMM to fold the next RMSNorm in (x larger than L2 keeps): 41412 x 520, a last column block of 8."""
    pair = wl.PairCfg("fold", wl.uniform_model(3, 520, 4, 2, 64, 128, 300), wl.uniform_model(3, 128, 2, 2, 64, 128, 300), (0, 1, 2))
    W = wl.make_weights(pair, seed=6, regime="fanin")
    lens = [500] * 82 + [412]
    pr = wl.custom_prompts(300, lens, seed=6)
    assert recorded_prefill(pair, lens, W).find("gemm_tc_kernelILi100E")
    s = make_session(pair, W, pr)
    try:
        ek, ev, el, tally = compare_prefill(s, pair, W, pr, seqs=[0, 41, 82])
        print(f"K {ek:.2e} V {ev:.2e} logits {el:.2e}")
        assert not tally.mismatches, tally.report()
    finally:
        s.close()
