"""What the base step's attention may meet in its inputs, whichever kernel serves it: cache rows at or beyond a sequence's length, which
are unspecified and here hold NaN.  First step and generation step, against the oracle on the cache that the GPU left."""
import numpy as np
import pytest

import workloads as wl
from parity_util import TOL, make_session, rel_fro
from recorded_graph import recorded_prefill
from test_step_mma_gpu import _step

pytestmark = pytest.mark.gpu


def _pair(hd, heads, d=264, ffn=520, dtype="bf16", qk_norm=False):
    return wl.PairCfg("values", wl.uniform_model(2, 128, 2, 1, hd, 128, 300, qk_norm), wl.uniform_model(2, d, heads[0], heads[1], hd, ffn, 300, qk_norm),
                      (0, 1), dtype=dtype)


def _compare(pair, W, lens, fill=None):
    """A first step and a generation step, each against the oracle's step over the cache that it has read."""
    import torch
    pr = wl.custom_prompts(300, lens, seed=6)
    s = make_session(pair, W, pr, extra_len=1)
    try:
        if fill is not None:
            for t in s.cache.k + s.cache.v:
                t.fill_(fill)
        logits, _ = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        toks, cur = [int(pr.seq(b)[-1]) for b in range(pr.batch)], list(lens)
        for step in range(2):
            logits = logits.cpu().numpy()
            for b in range(pr.batch):
                want = _step(pair, W, toks[b], [s.cache.gather(i, b, cur[b]) for i in range(2)])[0]
                assert rel_fro(logits[b], want) <= TOL[pair.dtype], f"step {step} sequence {b}"
            if step == 0:
                toks = [(7 * b + 5) % 300 for b in range(pr.batch)]
                logits, _ = s.decode_step(torch.tensor(toks, dtype=torch.int32, device=s.device), cur)
                s.poll()
                cur = [n + 1 for n in cur]
    finally:
        s.close()


@pytest.mark.parametrize("kernel,pair,lens", [
    ("step_attn_mma", _pair(64, (24, 8), 1544, 2568), [9, 130, 65]),              # the chain of three sequences
    ("step_attn_mma", _pair(64, (8, 2)), [1, 63, 64, 65, 200]),
    ("step_attn_mma", _pair(128, (6, 2), qk_norm=True), [15, 16, 17, 33, 118]),
    ("step_attn_mma", _pair(64, (4, 1)), [4101]),
    ("step_mega_mma", _pair(64, (8, 2)), [3, 100]),
    ("step_mega_kernel", _pair(32, (8, 2)), [3, 100]),
    ("step_attn_paged", _pair(32, (8, 2)), [1, 63, 64, 65, 200]),
    ("step_attn_kernel", _pair(24, (8, 2)), [1, 63, 64, 65, 200]),
    ("step_mega_kernel", _pair(64, (8, 2), dtype="f32"), [3, 100]),
    ("step_attn_paged", _pair(64, (8, 2), dtype="f32"), [1, 63, 64, 65, 200]),
], ids=str)
def test_rows_beyond_a_sequence_may_hold_anything(kernel, pair, lens):
    W = wl.make_weights(pair, seed=6, regime="fanin")
    assert recorded_prefill(pair, lens, W).find(kernel)
    _compare(pair, W, lens, fill=float("nan"))


@pytest.mark.parametrize("kernel,pair,lens", [
    ("step_attn_mma", _pair(64, (24, 8), 1544, 2568), [9, 130, 65]),
    ("step_attn_mma", _pair(64, (8, 2)), [1, 63, 64, 65, 200]),
    ("step_attn_mma", _pair(128, (6, 2)), [15, 16, 17, 33, 118]),
    ("step_mega_mma", _pair(64, (8, 2)), [3, 100]),
], ids=str)
@pytest.mark.parametrize("up", [-12, 0, 14, 17])
def test_queries_of_any_size(kernel, pair, lens, up):
    """Queries of 2^up times the ordinary size (up to about 4 x 2^up; halves end at 65504 and lose bits below 6e-5) on keys of 2^-up of it, so
    that the scores stay as they are; the cache is what the GPU holds, so that small keys are what they are."""
    W = wl.make_weights(pair, seed=6, regime="fanin")
    for i in range(2):
        W[f"base.L{i}.wq"] = W[f"base.L{i}.wq"] * np.float32(2.0 ** up)
        down = np.float32(2.0 ** min(12, -up))      # (keys of up to some thousand: halves, too)
        W[f"base.L{i}.wk"] = W[f"base.L{i}.wk"] * down
        W[f"pred.L{i}.fk"] = W[f"pred.L{i}.fk"] * down
    assert recorded_prefill(pair, lens, W).find(kernel)
    _compare(pair, W, lens)
