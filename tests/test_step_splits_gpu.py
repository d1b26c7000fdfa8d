"""Key-range splits of the CUDA-core persistent step kernel (fp32 mode, and 16-bit mode with narrow heads) on models whose layers
differ in kv heads: a layer's split count goes by its own kv heads, so that its partial results fit their buffer.  The bytes behind
the workspace are checked too."""
import numpy as np
import pytest

import workloads as wl
from oracle import kvp_oracle as orc
from parity_util import TOL, make_session, rel_fro
from recorded_graph import Recorded, recorded_prefill

pytestmark = pytest.mark.gpu
TAIL = 1 << 20


@pytest.mark.parametrize("dtype,hd,lens", [("f32", 16, [700, 650, 1, 699]), ("f32", 32, [1300, 1281]), ("bf16", 32, [700, 64, 641])], ids=str)
def test_splits_of_layers_with_few_and_many_kv_heads(dtype, hd, lens):
    import torch
    base = wl.ModelCfg(64, 97, tuple(wl.LayerCfg(n, n, hd, 96) for n in (1, 16, 1, 12)))
    pair = wl.PairCfg("few_many", wl.uniform_model(2, 64, 2, 1, hd, 96, 97), base, (0, 0, 1, 1), dtype=dtype)
    W = wl.make_weights(pair, seed=11, regime="fanin")
    pr = wl.custom_prompts(97, lens, seed=11)
    s = make_session(pair, W, pr, extra_len=2)
    n = s.workspace.numel()
    whole = torch.full((n + TAIL,), 0xA5, dtype=torch.uint8, device=s.device)
    whole[:n] = 0
    s.workspace = whole[:n]
    torch.cuda.synchronize()
    tol = TOL[dtype]
    try:
        logits, _ = s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        logits = logits.cpu().numpy()
        ref = orc.prefill_predict(pair, W, pr)
        caches = {b: ref[b][0] for b in range(pr.batch)}
        for b in range(pr.batch):
            assert rel_fro(logits[b], ref[b][1]) <= tol
        # the step's own workspace is smaller than the prefill's: a view that ends where it ends
        import paper_2410_08391_b200 as kvp
        n = kvp.kvp_workspace_bytes(s.h, len(lens), len(lens))
        whole[n:] = 0xA5
        s.workspace = whole[:n]
        cur, g = list(lens), np.random.default_rng(5)
        for _ in range(2):
            nxt = g.integers(0, 97, size=pr.batch).astype(np.int32)
            logits, tok = s.decode_step(torch.from_numpy(nxt).to(s.device), cur)
            s.poll()
            logits, cur = logits.cpu().numpy(), [c + 1 for c in cur]
            for b in range(pr.batch):
                want, caches[b] = orc.decode_step(pair, W, int(nxt[b]), caches[b])
                assert rel_fro(logits[b], want) <= tol
        assert bool((whole[n:] == 0xA5).all()), "bytes behind the workspace were written"
    finally:
        s.close()


@pytest.mark.parametrize("lens,ctas", [([64], 43), ([300], 43), ([999], 64), ([300] * 4, 80), ([3999], 148)], ids=str)
def test_every_attention_item_of_a_step_has_a_cta(lens, ctas):
    """A small model takes fewer CTAs than there are SMs (16 rows of its widest projection each: 688 / 16), but a key range of a
    sequence and kv head is not left to a second round while SMs are free."""
    import torch

    import paper_2410_08391_b200 as kvp
    pair = wl.pair("c1")
    s = make_session(pair, wl.make_weights(pair, seed=1), wl.custom_prompts(pair.base.vocab, lens, seed=1), extra_len=1)
    try:
        tok = torch.zeros(len(lens), dtype=torch.int32, device=s.device)
        g = Recorded(s, lambda: kvp.kvp_decode_step(s.h, tok, lens, s.cache, s.workspace, s.logits, s.first, s.stream))
        assert g.grids("step_mega_kernel") == [(ctas, 1, 1)]
    finally:
        s.close()


@pytest.mark.parametrize("lens,ctas", [([64], 43), ([999], 64), ([300] * 4, 64), ([3999], 72)], ids=str)
def test_every_attention_item_of_a_piece_has_a_cta(lens, ctas):
    """The same beside a prefill, where the pieces take at most 72 SMs and the key ranges go by that."""
    grids = recorded_prefill(wl.pair("c1"), lens).grids("step_mega_kernel")
    assert len(grids) == 2 and all(g == (ctas, 1, 1) for g in grids)
