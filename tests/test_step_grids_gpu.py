"""How many CTAs the step's tensor-core projections take: two an SM up to 64 sequences, one from 65 on, where two accumulators fill an SM's
tensor memory.  Read from a recorded generation step, with its results against the oracle at sizes around both lines of the rule."""
import numpy as np
import pytest

import workloads as wl
from parity_util import TOL, make_session, rel_fro
from recorded_graph import Recorded
from test_step_mma_gpu import _step

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("batch,ctas", [(64, 296), (65, 148), (72, 148), (83, 148), (128, 148)])
def test_one_cta_an_sm_where_two_do_not_fit_its_tensor_memory(batch, ctas):
    import torch

    import paper_2410_08391_b200 as kvp
    # gate and up: 320 tiles of 8 k blocks, at least 8 of them a CTA
    pair = wl.PairCfg("grids", wl.uniform_model(1, 64, 1, 1, 64, 64, 300), wl.uniform_model(1, 512, 4, 2, 64, 20480, 300), (0,))
    W = wl.make_weights(pair, seed=3, regime="fanin")
    lens = [1 + (7 * b) % 70 for b in range(batch)]
    pr = wl.custom_prompts(300, lens, seed=3)
    s = make_session(pair, W, pr, extra_len=1)
    try:
        s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), lens)
        s.poll()
        toks = (np.arange(batch) * 5 + 3) % 300
        dev = torch.tensor(toks, dtype=torch.int32, device=s.device)
        grids = Recorded(s, lambda: kvp.kvp_decode_step(s.h, dev, lens, s.cache, s.workspace, s.logits, s.first, s.stream)).grids("step_gemm_kernel")
        assert max(g[0] for g in grids) == ctas
        logits, _ = s.decode_step(dev, lens)
        s.poll()
        logits = logits.cpu().numpy()
        for b in (0, 7, 8, 63, batch - 1):
            want = _step(pair, W, int(toks[b]), [s.cache.gather(0, b, lens[b] + 1)])[0]
            assert rel_fro(logits[b], want) <= TOL["bf16"]
    finally:
        s.close()
