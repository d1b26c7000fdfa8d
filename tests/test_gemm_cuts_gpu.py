"""The tensor-core GEMM at every tile width and both ways of cutting the work: rows, columns and k that leave the last tile, the last
piece of a cache row and the last k block ragged, against the oracle.  Which width and cut a call takes is the launcher's rule; the
recorded graph says that it is the one meant here."""
import re

import pytest

import workloads as wl
from parity_util import TOL, assert_first_tokens, compare_prefill, make_session
from recorded_graph import recorded_prefill

pytestmark = pytest.mark.gpu
TWO = [1000, 999]                # 1999 rows = 15.6 row blocks, on 100 SMs beside the step's 48
SIX = [301, 200, 190, 64, 35, 1000]      # 1790 rows = 14 row blocks, on 148


def _launches(g, epilogue):
    """(tile width, CTAs) of the GEMMs with this epilogue, in order"""
    found = [(int(re.search("gemm_tc_kernelILi%dELi(\\d+)E" % epilogue, g.name[x]).group(1)), g.grid[x][0]) for x in sorted(
        g.find("gemm_tc_kernelILi%dE" % epilogue), key=lambda x: len(g.before(x)))]
    return found


# residual: O and down projection of the first layer, (width, CTAs): whole tiles take a CTA each here, shares of the k blocks every SM;
# widths of its QKV projection and of its predictor
@pytest.mark.parametrize("d,ffn,heads,base_kv,lens,residual,qkv,predictor", [
    (72, 128, (1, 1), 1, [70], [(128, 1), (128, 1)], 128, 128),                         # one ragged tile
    (264, 2056, (2, 2), 2, TWO, [(128, 48), (128, 100)], 128, 128),                     # down: 33 k blocks of 48 tiles, shared by 100 CTAs
    (520, 4104, (2, 2), 2, TWO, [(128, 80), (256, 100)], 128, 128),                     # shares of 256-wide tiles, the last of 8 columns
    (840, 200, (3, 1), 2, TWO, [(160, 96), (160, 96)], 128, 128),                       # 5.25 tiles
    (1032, 136, (10, 2), 13, TWO, [(192, 96), (192, 96)], 192, 192),                    # 5.4; 896 = 4.7 x 192; 832 = 4.3 x 192
    (1224, 72, (3, 3), 3, TWO, [(224, 96), (224, 96)], 128, 128),                       # 5.5
    (1368, 64, (15, 3), 19, TWO, [(256, 96), (256, 96)], 256, 256),                     # 5.3; 1344 = 5.25 x 256; 1216 = 4.75 x 256
    (1032, 4104, (4, 1), 9, SIX, [(128, 126), (256, 148)], 128, 128),                   # 148 SMs, shares of 256-wide tiles
], ids=str)
def test_every_cut_matches_oracle(d, ffn, heads, base_kv, lens, residual, qkv, predictor):
    aux = wl.uniform_model(2, d, heads[0], heads[1], 64, ffn, 500)
    pair = wl.PairCfg("cuts", aux, wl.uniform_model(2, 128, base_kv, base_kv, 64, 128, 500), (0, 1))
    W = wl.make_weights(pair, seed=6, regime="fanin")
    g = recorded_prefill(pair, lens, W)
    assert _launches(g, 1) == residual and _launches(g, 3)[0][0] == qkv and {w for w, _ in _launches(g, 4)} == {predictor}
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


def _pairs(g, epilogue):
    return len(g.find("gemm_tc_kernelILi%dELi256ELb1E" % epilogue))


# More than 4096 tokens (with fewer, other streams run beside the GEMMs and single CTAs take them).  4300 rows: the second CTA of the last
# pair has 76 of its 128; 4168 and 5200: none.  1544 columns: 6 x 256 + 8, 24 k blocks + 8.
# epilogues that run in pairs: 1 residual (in shares of the k blocks), 2 gate / up, 3 QKV, 100 residual with the norm folded in
@pytest.mark.parametrize("d,ffn,heads,hd,lens,pairs", [
    (1544, 4160, (24, 3), 128, [850] * 5 + [50], (1, 2, 3)),
    (1544, 4160, (24, 3), 128, [833] * 5 + [3], (1, 2, 3)),
    (2312, 2112, (24, 3), 128, [1008] * 5 + [100, 60], (2, 3, 100)),
], ids=str)
def test_cta_pairs_match_oracle(d, ffn, heads, hd, lens, pairs):
    pair = wl.PairCfg("pairs", wl.uniform_model(2, d, heads[0], heads[1], hd, ffn, 300), wl.uniform_model(2, 128, 2, 2, 64, 128, 300), (0, 1))
    W = wl.make_weights(pair, seed=8, regime="fanin")
    g = recorded_prefill(pair, lens, W)
    assert not any(_pairs(recorded_prefill(pair, [500] * 6, W), e) for e in (1, 2, 3, 100))
    assert tuple(e for e in (1, 2, 3, 100) if _pairs(g, e)) == pairs
    pr = wl.custom_prompts(300, lens, seed=8)
    s = make_session(pair, W, pr)
    try:
        ek, ev, el, tally = compare_prefill(s, pair, W, pr, seqs=[0, len(lens) - 2, len(lens) - 1])
        print(f"K {ek:.2e} V {ev:.2e} logits {el:.2e}")
        assert_first_tokens(tally, TOL[pair.dtype], "pairs")
    finally:
        s.close()
