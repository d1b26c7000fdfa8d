"""The persistent tensor-core step kernel (16-bit weights, batch <= 4) at the sizes where its tiling can go wrong: several
groups of tiles per CTA (vocabulary), chunks of K with a ragged end, fewer outputs than CTAs, key ranges over several pages
and items, a new key that opens a page; first step and generation steps, against the oracle."""
import numpy as np
import pytest

import workloads as wl
from oracle import kvp_oracle as orc
from parity_util import TOL, make_session, rel_fro

pytestmark = pytest.mark.gpu


def _pair(name):
    if name == "wide":       # 20 000 / 148 = 136 head rows per CTA (2 groups of tiles); K = 520 and 4136: no multiples of 64
        return wl.PairCfg(name, wl.uniform_model(2, 192, 4, 1, 64, 320, 20000), wl.uniform_model(3, 520, 8, 2, 64, 4136, 20000), (0, 1, 1))
    if name == "hd128":      # head_dim 128, 8 query heads per kv head, query / key norm, K = 1032
        return wl.PairCfg(name, wl.uniform_model(2, 256, 2, 1, 128, 512, 1000, qk_norm=True),
                          wl.uniform_model(2, 1032, 8, 1, 128, 2056, 1000, qk_norm=True), (0, 1))
    # more (sequence, kv head) pairs than CTAs can split: one split per item; layers of different widths
    return wl.PairCfg(name, wl.uniform_model(2, 192, 4, 1, 64, 320, 1000), wl.uniform_model(2, 256, 48, 48, 64, 192, 1000), (0, 1))


@pytest.mark.parametrize("name,lens", [("wide", [1]), ("wide", [64, 191]), ("wide", [130, 64, 3]), ("hd128", [700]),
                                       ("hd128", [63, 320, 1, 65]), ("many", [200, 64, 65, 129])], ids=str)
def test_small_batch_steps_match_oracle(name, lens):
    import torch
    pair = _pair(name)
    W = wl.make_weights(pair, seed=3, regime="fanin")
    pr = wl.custom_prompts(pair.base.vocab, lens, seed=3)
    s = make_session(pair, W, pr, extra_len=2)
    tol = TOL[pair.dtype]      # the parity tolerance of the 16-bit mode: the predicted cache in front of the step is 16-bit
    try:
        logits, _ = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        logits = logits.cpu().numpy()
        ref = orc.prefill_predict(pair, W, pr)
        caches = {b: ref[b][0] for b in range(pr.batch)}
        for b in range(pr.batch):
            assert rel_fro(logits[b], ref[b][1]) <= tol
        cur, g = list(lens), np.random.default_rng(5)
        for _ in range(2):
            nxt = g.integers(0, pair.base.vocab, size=pr.batch).astype(np.int32)
            logits, tok = s.decode_step(torch.from_numpy(nxt).to(s.device), cur)
            s.poll()
            logits, cur = logits.cpu().numpy(), [c + 1 for c in cur]
            assert s.cache.seq_lens[:pr.batch].cpu().tolist() == cur
            for b in range(pr.batch):
                want, caches[b] = orc.decode_step(pair, W, int(nxt[b]), caches[b])
                assert rel_fro(logits[b], want) <= tol
                assert int(tok[b]) == int(np.argmax(logits[b]))
                for i in range(pair.base.n_layers):
                    k, v = s.cache.gather(i, b, cur[b])
                    assert rel_fro(k[-1], caches[b][i][0][-1]) <= tol and rel_fro(v[-1], caches[b][i][1][-1]) <= tol
    finally:
        s.close()
