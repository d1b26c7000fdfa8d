"""The base step as a chain of launches (more than 4 sequences, or long caches), whose attention appends the step's own key and value
and writes the next projection's operand rows: batches at the edges of the groups of 8 rows, outputs and widths that leave tiles
ragged, layers of different widths, new keys that open a page, end it, or lie in the last of several key ranges, every ring depth."""
import numpy as np
import pytest

import workloads as wl
from oracle import kvp_oracle as orc
from parity_util import TOL, make_session, rel_fro
from test_step_mma_gpu import _step, _two_terms

pytestmark = pytest.mark.gpu


def _pair(name):
    if name == "wide":       # K = 520 and 4136: no multiples of 64
        return wl.PairCfg(name, wl.uniform_model(2, 192, 4, 1, 64, 320, 3001), wl.uniform_model(3, 520, 8, 2, 64, 4136, 3001), (0, 1, 1))
    if name == "hd128":      # head_dim 128, 8 query heads per kv head, query / key norm
        return wl.PairCfg(name, wl.uniform_model(2, 256, 2, 1, 128, 512, 1000, qk_norm=True),
                          wl.uniform_model(2, 1032, 8, 1, 128, 2112, 1000, qk_norm=True), (0, 1))
    if name == "small":      # one tile, or less, per projection
        return wl.PairCfg(name, wl.uniform_model(2, 64, 2, 1, 64, 128, 67), wl.uniform_model(3, 72, 1, 1, 64, 72, 67), (0, 1, 1))
    if name == "mixed":      # layers that differ in heads and FFN width
        layers = tuple(wl.LayerCfg(2 * n, n, 64, f) for n, f in ((1, 64), (3, 200), (2, 136)))
        return wl.PairCfg(name, wl.uniform_model(2, 64, 2, 1, 64, 128, 131), wl.ModelCfg(136, 131, layers), (0, 1, 1))
    return wl.PairCfg(name, wl.uniform_model(2, 64, 2, 1, 32, 128, 131), wl.uniform_model(2, 128, 4, 2, 32, 128, 131), (0, 1))   # hd32


CASES = [("wide", [64, 1, 30, 127, 128]), ("wide", [3 + i for i in range(33)]), ("hd128", [65, 2, 129, 64, 63, 1, 320, 700, 5]), ("small", [5, 63, 64, 65, 1]),
         ("small", [1 + i % 9 for i in range(64)]), ("small", [1 + i % 70 for i in range(65)]), ("small", [2 + i % 5 for i in range(128)]),
         ("mixed", [64, 9, 128, 3, 77, 191]), ("hd32", [64, 9, 70, 3, 77, 63]), ("small", [4200]), ("hd128", [4160, 4223, 64])]


@pytest.mark.parametrize("name,lens", CASES, ids=lambda v: str(v).replace(" ", "")[:30])
def test_chain_matches_oracle(name, lens):
    """The step alone, on the cache that it reads: its activations enter as two bf16 terms (16 bits), whose rounding moves the oracle by
    e2; the kernel's own rounding is another draw of the same size, and its sums lose at most 2^-23 of themselves with each of the
    K / 16 instructions they go through."""
    import torch
    pair = _pair(name)
    W = wl.make_weights(pair, seed=3, regime="fanin")
    pr = wl.custom_prompts(pair.base.vocab, lens, seed=3)
    s = make_session(pair, W, pr, extra_len=2)
    k_max = max([pair.base.d_model] + [c.ffn_dim for c in pair.base.layers] + [c.d_q for c in pair.base.layers])
    seen = range(pr.batch) if pr.batch <= 9 else sorted({0, 3, 7, 31, 32, pr.batch - 2, pr.batch - 1} & set(range(pr.batch)))
    try:
        logits, _ = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        logits = logits.cpu().numpy()
        cur, g = list(lens), np.random.default_rng(5)
        toks = [int(pr.seq(b)[-1]) for b in range(pr.batch)]
        for step in range(3):      # the first step, then two generation steps
            for b in seen:
                cache = [s.cache.gather(i, b, cur[b]) for i in range(pair.base.n_layers)]
                want, rows = _step(pair, W, toks[b], cache)
                e2 = rel_fro(_step(pair, W, toks[b], cache, _two_terms)[0], want)
                err = rel_fro(logits[b], want)
                assert err <= 2 * e2 + k_max / 16 * 2.0 ** -23, f"step {step} sequence {b}: {err:.2e}, two terms {e2:.2e}"
                for i in range(pair.base.n_layers if step else 0):
                    for got, ref in zip(cache[i], rows[i]):      # a half, and what the two terms in front of it leave of the row's rms
                        lim = 2.0 ** -11 * (np.abs(ref) + np.sqrt(np.mean(ref * ref)))
                        assert np.all(np.abs(got[-1] - ref) <= lim), f"step {step} sequence {b} layer {i}"
            if step == 2:
                break
            toks = [int(t) for t in g.integers(0, pair.base.vocab, size=pr.batch)]
            logits, tok = s.decode_step(torch.tensor(toks, dtype=torch.int32, device=s.device), cur)
            s.poll()
            logits, cur = logits.cpu().numpy(), [c + 1 for c in cur]
            assert s.cache.seq_lens[:pr.batch].cpu().tolist() == cur
            assert [int(t) for t in tok.cpu()] == [int(np.argmax(r)) for r in logits]
    finally:
        s.close()
