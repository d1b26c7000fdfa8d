"""The persistent step kernel of the fp32 mode at widths of a head group where its attention gives threads different work: a value sum by
heads (head_dim 128 with 3 heads or more to a kv head, 64 with 5 or more) and by keys, groups that leave threads without a share, one and
several key ranges; first step and generation steps against the oracle (fp32 products in another order: 1e-4)."""
import numpy as np
import pytest

import workloads as wl
from oracle import kvp_oracle as orc
from parity_util import TOL, make_session, rel_fro
from recorded_graph import recorded_prefill

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hd,heads,lens,qk_norm", [
    (128, (6, 2), [70], False), (128, (6, 2), [1, 64, 65, 400], True), (128, (8, 1), [130, 63], False), (128, (5, 1), [300], True),
    (64, (10, 2), [64, 1, 200], False), (64, (6, 1), [129], True), (64, (7, 1), [900, 5], False), (64, (8, 1), [63, 64], True),
    (32, (7, 1), [66, 3], False), (16, (3, 1), [130], False), (16, (14, 2), [9, 64, 65, 300], True), (16, (5, 1), [700], False),
], ids=str)
def test_head_groups_match_oracle(hd, heads, lens, qk_norm):
    import torch
    pair = wl.PairCfg("groups", wl.uniform_model(2, 64, 2, 1, hd, 96, 211, qk_norm), wl.uniform_model(2, 152, heads[0], heads[1], hd, 264, 211, qk_norm),
                      (0, 1), dtype="f32")
    W = wl.make_weights(pair, seed=5, regime="fanin")
    assert recorded_prefill(pair, lens, W).find("step_mega_kernel")
    pr = wl.custom_prompts(211, lens, seed=5)
    s = make_session(pair, W, pr, extra_len=2)
    tol = TOL["f32"]
    try:
        logits, _ = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        logits = logits.cpu().numpy()
        ref = orc.prefill_predict(pair, W, pr)
        caches = {b: ref[b][0] for b in range(pr.batch)}
        for b in range(pr.batch):
            assert rel_fro(logits[b], ref[b][1]) <= tol
        cur = list(lens)
        for step in range(2):
            nxt = np.array([(31 * b + 17 * step + 3) % 211 for b in range(pr.batch)], np.int32)
            logits, _ = s.decode_step(torch.from_numpy(nxt).to(s.device), cur)
            s.poll()
            logits, cur = logits.cpu().numpy(), [c + 1 for c in cur]
            for b in range(pr.batch):
                want, caches[b] = orc.decode_step(pair, W, int(nxt[b]), caches[b])
                assert rel_fro(logits[b], want) <= tol
                for i in range(2):
                    k, v = s.cache.gather(i, b, cur[b])
                    assert rel_fro(k[-1], caches[b][i][0][-1]) <= tol and rel_fro(v[-1], caches[b][i][1][-1]) <= tol
    finally:
        s.close()
