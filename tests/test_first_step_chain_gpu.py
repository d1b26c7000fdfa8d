"""First steps of three and four sequences as a chain of launches (three bf16 terms an activation): rows and columns that
leave the last weight tile ragged, k ranges of one k block and of more than eight, beside the prefill and behind it.  Against the oracle, and
the step alone, on the GPU's own cache: a quarter of what dropping the third term moves the oracle bounds its error (sums of up to eight k
blocks go through few instructions that round towards zero, and partial sums are added in fp32)."""
import numpy as np
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


def _pair(hd, heads, d, ffn, n, qk_norm=False):
    return wl.PairCfg("chain3", wl.uniform_model(2, 128, 2, 1, hd, 128, 300, qk_norm), wl.uniform_model(n, d, heads[0], heads[1], hd, ffn, 300, qk_norm),
                      (0,) * (n // 2) + (1,) * (n - n // 2))


@pytest.mark.parametrize("pair,lens", [
    (_pair(128, (24, 6), 3072, 8192, 4), [33, 70, 5]),                     # k ranges of up to 128 blocks, up to 24 partial sums an output
    (_pair(128, (16, 4), 2056, 8200, 6), [33, 70, 5]),
    (_pair(64, (16, 4), 1544, 8200, 4, qk_norm=True), [20, 3, 64, 40]),
], ids=str)
def test_the_chain_is_as_exact_as_the_persistent_kernel(pair, lens):
    """Both serve the same call, the chain from device memory and the persistent kernel from host memory: on the same cache the chain's
    logits are no further from 64 bits (0.74 to 0.85 of the other's distance, 0.02 of it by the order of the partial sums)."""
    import torch

    import paper_2410_08391_b200 as kvp
    W = wl.make_weights(pair, seed=9, regime="fanin")
    assert recorded_prefill(pair, lens, W).find("step_gemm_kernel")
    pr = wl.custom_prompts(300, lens, seed=9)
    s = make_session(pair, W, pr)
    try:
        logits, _ = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        logits = logits.cpu().numpy()
        host, first = torch.zeros((len(lens), 300)).pin_memory(), torch.zeros(len(lens), dtype=torch.int32).pin_memory()
        n0 = kvp.kvp_launch_count(s.h)
        kvp.kvp_prefill_predict_host(s.h, torch.from_numpy(pr.tokens).pin_memory(), lens, s.cache, s.workspace, s.logits, host, first, s.stream)
        s.poll()
        assert kvp.kvp_launch_count(s.h) - n0 < 5 * pair.base.n_layers + 40      # (no chain: that is eight launches a base layer alone)
        want = [_step(pair, W, int(pr.seq(b)[-1]), [s.cache.gather(i, b, n) for i in range(pair.base.n_layers)])[0] for b, n in enumerate(lens)]
        rms = lambda got: float(np.sqrt(np.mean([rel_fro(got[b], want[b]) ** 2 for b in range(len(lens))])))  # noqa: E731
        chain, persistent = rms(logits), rms(host.numpy())
        print(f"chain {chain:.2e}, persistent kernel {persistent:.2e}")
        assert chain <= persistent
    finally:
        s.close()


@pytest.mark.parametrize("lens", [[20], [20, 9]], ids=str)
def test_one_and_two_sequences_stay_with_the_persistent_kernel(lens):
    """It is the more exact one for them, however many weights a layer has (here 193 MB) and however short the prompt."""
    pair = wl.PairCfg("large_layer", wl.uniform_model(1, 64, 1, 1, 128, 64, 300), wl.uniform_model(1, 4104, 8, 2, 128, 7176, 300), (0,))
    g = recorded_prefill(pair, lens)
    assert g.find("step_mega_mma_kernel") and not g.find("step_gemm_kernel")
