"""The persistent tensor-core step kernel (16-bit weights, batch <= 4) at the sizes where its tiling can go wrong: several
groups of tiles per CTA (vocabulary, residual stream), chunks of K with a ragged end, fewer outputs than CTAs, every width of a
head group, key ranges over several pages and items, a new key that opens a page; first step and generation steps, against the
oracle.  End to end at the parity tolerance, and the step alone, on the GPU's own cache, at fp32 accuracy."""
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
    if name == "small":      # fewer outputs than CTAs (148, or the 72 of a piece) in every projection and the head
        return wl.PairCfg(name, wl.uniform_model(2, 64, 2, 1, 64, 128, 67), wl.uniform_model(3, 72, 1, 1, 64, 64, 67), (0, 1, 1))
    if name == "deep":       # 12 000 / 148 = 82 residual rows per CTA: a second group of tiles
        return wl.PairCfg(name, wl.uniform_model(1, 64, 2, 1, 64, 128, 300), wl.uniform_model(1, 12000, 2, 1, 64, 64, 300), (0,))
    if name.startswith("g"):     # g<query heads per kv head>x<head_dim>
        g, hd = (int(n) for n in name[1:].split("x"))
        return wl.PairCfg(name, wl.uniform_model(2, 192, 2, 1, hd, 320, 500), wl.uniform_model(2, 264, 2 * g, 2, hd, 520, 500), (0, 1))
    if name == "kv4x128":    # a long cache is more pages than CTAs: several pages a key range, through one page slot
        return wl.PairCfg(name, wl.uniform_model(2, 192, 2, 1, 128, 320, 500), wl.uniform_model(2, 264, 8, 4, 128, 520, 500), (0, 1))
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


def _two_terms(x):
    """What the first two of the kernel's three bf16 terms hold of x."""
    hi = wl.round_to_bf16(x.astype(np.float32)).astype(np.float64)
    return hi + wl.round_to_bf16((x - hi).astype(np.float32)).astype(np.float64)


def _step(pair, W, token, cache, cut=lambda v: v):
    """One base step at the position of the cache's last row, whose key and value are in the cache already (in a first step they
    are predicted, in a generation step the step's own).  `cut`: applied to every projection's input.
    Returns the logits and, per layer, the key and the value that the step itself computes for its position."""
    cfg, n = pair.base, cache[0][0].shape[0]
    pos = np.array([n - 1])
    x = W["base.embed"][[token]].astype(np.float64)
    rows = []
    for i, c in enumerate(cfg.layers):
        b = f"base.L{i}."
        w = lambda leaf: W[b + leaf].astype(np.float64)  # noqa: E731
        h = cut(orc.rmsnorm(x, W[b + "attn_norm"], cfg.rms_eps))
        q = (h @ w("wq").T).reshape(1, c.n_q_heads, c.head_dim)
        k = (h @ w("wk").T).reshape(1, c.n_kv_heads, c.head_dim)
        q, k = orc.qk_norm(cfg, W, b, q, k)
        rows.append((orc.rope(k, pos, cfg.rope_theta).reshape(-1), (h @ w("wv").T).reshape(-1)))
        kc, vc = (a.astype(np.float64).reshape(n, c.n_kv_heads, c.head_dim) for a in cache[i])
        a = orc.attention(orc.rope(q, pos, cfg.rope_theta), kc, vc, pos)
        x = x + cut(a.reshape(1, -1)) @ w("wo").T
        h = cut(orc.rmsnorm(x, W[b + "ffn_norm"], cfg.rms_eps))
        x = x + cut(orc.silu(h @ w("w_gate").T) * (h @ w("w_up").T)) @ w("w_down").T
    return (cut(orc.rmsnorm(x, W["base.final_norm"], cfg.rms_eps)) @ W["base.lm_head"].astype(np.float64).T)[0], rows


ALONE = [("wide", [1]), ("wide", [64, 191]), ("wide", [130, 64, 3]), ("hd128", [700]), ("hd128", [321, 64]), ("hd128", [63, 320, 1, 65]),
         ("many", [200, 64, 65, 129]), ("small", [70]), ("small", [5, 127]), ("small", [64, 1, 300]), ("small", [130, 63, 64, 65]),
         ("deep", [70]), ("deep", [65, 3]), ("deep", [64, 5, 9, 130]), ("g5x64", [200]), ("g6x64", [66, 300]), ("g7x64", [3, 64, 190]),
         ("g8x64", [127, 64, 1, 320]), ("g1x128", [130]), ("g3x128", [63, 200]), ("g5x128", [300, 64]), ("g8x128", [65, 2, 129]),
         ("kv4x128", [4000]), ("kv4x128", [1990, 2050]), ("g8x128", [4030, 3900])]


@pytest.mark.parametrize("name,lens", ALONE, ids=str)
def test_step_alone_keeps_every_term(name, lens):
    """The step on the cache that it reads, taken back from the GPU: no rounding of the cache is left in the comparison, only the
    kernel's own.  Its activations enter as three bf16 terms (24 bits); with the last term dropped the oracle itself moves by
    `e2`.  An eighth of that bounds what the logits may be off; a quarter for rows of more than 8192, whose sums go through more
    than 16 instructions that round towards zero.  A new key or value is one IEEE half: 2^-11 of itself,
    and the same share of the row's rms for what the fp32 arithmetic in front of it adds."""
    import torch
    pair = _pair(name)
    W = wl.make_weights(pair, seed=3, regime="fanin")
    pr = wl.custom_prompts(pair.base.vocab, lens, seed=3)
    s = make_session(pair, W, pr, extra_len=2)
    share = 0.125 if pair.base.d_model <= 8192 else 0.25
    try:
        logits, _ = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        logits = logits.cpu().numpy()
        cur, g = list(lens), np.random.default_rng(5)
        toks = [int(pr.seq(b)[-1]) for b in range(pr.batch)]
        worst = 0.0
        for step in range(3):      # the first step, then two generation steps
            for b in range(pr.batch):
                cache = [s.cache.gather(i, b, cur[b]) for i in range(pair.base.n_layers)]
                want, rows = _step(pair, W, toks[b], cache)
                e2 = rel_fro(_step(pair, W, toks[b], cache, _two_terms)[0], want)
                err = rel_fro(logits[b], want)
                worst = max(worst, err / e2)
                assert err <= share * e2, f"step {step} sequence {b}: {err:.2e}, two terms {e2:.2e}"
                for i in range(pair.base.n_layers if step else 0):
                    for got, ref in zip(cache[i], rows[i]):
                        lim = 2.0 ** -11 * (np.abs(ref) + np.sqrt(np.mean(ref * ref)))
                        assert np.all(np.abs(got[-1] - ref) <= lim), f"step {step} sequence {b} layer {i}"
            if step == 2:
                break
            toks = [int(t) for t in g.integers(0, pair.base.vocab, size=pr.batch)]
            logits, _ = s.decode_step(torch.tensor(toks, dtype=torch.int32, device=s.device), cur)
            s.poll()
            logits, cur = logits.cpu().numpy(), [c + 1 for c in cur]
        print(f"worst error / error of two terms: {worst:.3f}")
    finally:
        s.close()
