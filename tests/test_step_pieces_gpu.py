"""How many SMs the base step's pieces take beside the prefill of up to 4 sequences: few where the prefill lasts much longer, none (the
step runs after it, as one kernel) where it is over long before the step and the caller waits.  Read from the recorded graph and from
the number of launches, with the results of each against the oracle."""
import numpy as np
import pytest

import workloads as wl
from oracle import kvp_oracle as orc
from parity_util import TOL, make_session, rel_fro, run_prefill
from recorded_graph import recorded_prefill

pytestmark = pytest.mark.gpu


def test_a_long_prefill_leaves_the_pieces_few_sms():
    grids = recorded_prefill(wl.pair("t_small"), [150, 37, 1, 64]).grids("step_mega_mma_kernel")
    assert sorted(grids) == [(48, 1, 1)] * 2 + [(148, 1, 1)]      # a piece per auxiliary layer, the last one when the prefill is over


def test_a_step_that_is_the_longer_one_runs_in_pieces_or_after_the_prefill():
    """About 0.5 GB of base weights behind two narrow auxiliary layers: the prefill is estimated at 0.45 of the step."""
    import torch

    import paper_2410_08391_b200 as kvp
    pair = wl.PairCfg("wide_base", wl.uniform_model(2, 64, 2, 1, 64, 128, 500), wl.uniform_model(10, 1024, 8, 2, 64, 8192, 500), (0,) * 5 + (1,) * 5)
    W = wl.make_weights(pair, seed=4, regime="fanin")
    lens = [5, 3]
    pr = wl.custom_prompts(500, lens, seed=4)
    assert sorted(recorded_prefill(pair, lens, W).grids("step_mega_mma_kernel")) == [(72, 1, 1), (148, 1, 1)]
    ref = orc.prefill_predict(pair, W, pr)
    s = make_session(pair, W, pr)
    try:
        n0 = kvp.kvp_launch_count(s.h)
        logits, _ = run_prefill(s, pr)
        n1 = kvp.kvp_launch_count(s.h)
        host = torch.zeros((2, 500)).pin_memory()
        first = torch.zeros(2, dtype=torch.int32).pin_memory()
        kvp.kvp_prefill_predict_host(s.h, torch.from_numpy(pr.tokens).pin_memory(), lens, s.cache, s.workspace, s.logits, host, first, s.stream)
        s.poll()
        assert kvp.kvp_launch_count(s.h) - n1 == n1 - n0 - 1      # one step kernel instead of two pieces
        for b in range(2):
            assert rel_fro(logits[b], ref[b][1]) <= TOL["bf16"] and rel_fro(host[b].numpy(), ref[b][1]) <= TOL["bf16"]
            assert int(first[b]) == int(np.argmax(host[b].numpy()))
            for i in (0, 4, 5, 9):
                k, v = s.cache.gather(i, b, lens[b])
                assert rel_fro(k, ref[b][0][i][0]) <= TOL["bf16"] and rel_fro(v, ref[b][0][i][1]) <= TOL["bf16"]
    finally:
        s.close()


def test_the_last_layers_of_a_caller_that_waits_are_one_piece_on_all_sms():
    """The prefill is estimated at 1.1 of the step (4 layers of 36 us, 0.42 GB of base weights): its pieces reach some of the base layers
    meanwhile, and what is left is one launch.  Other callers get a piece per auxiliary layer."""
    import torch

    import paper_2410_08391_b200 as kvp
    n = 4
    pair = wl.PairCfg("waits", wl.uniform_model(n, 64, 2, 1, 64, 128, 500), wl.uniform_model(2 * n, 1024, 8, 2, 64, 8192, 500), tuple(i // 2 for i in range(2 * n)))
    W = wl.make_weights(pair, seed=4, regime="fanin")
    lens = [7]
    pr = wl.custom_prompts(500, lens, seed=4)
    ref = orc.prefill_predict(pair, W, pr)
    assert len(recorded_prefill(pair, lens, W).grids("step_mega_mma_kernel")) == n
    s = make_session(pair, W, pr)
    try:
        n0 = kvp.kvp_launch_count(s.h)
        logits, _ = run_prefill(s, pr)
        n1 = kvp.kvp_launch_count(s.h)
        host, first = torch.zeros((1, 500)).pin_memory(), torch.zeros(1, dtype=torch.int32).pin_memory()
        kvp.kvp_prefill_predict_host(s.h, torch.from_numpy(pr.tokens).pin_memory(), lens, s.cache, s.workspace, s.logits, host, first, s.stream)
        s.poll()
        fewer = (n1 - n0) - (kvp.kvp_launch_count(s.h) - n1)
        assert 1 <= fewer < n - 1
        assert rel_fro(logits[0], ref[0][1]) <= TOL["bf16"] and rel_fro(host[0].numpy(), ref[0][1]) <= TOL["bf16"]
        for i in (0, n, 2 * n - 1):
            k, v = s.cache.gather(i, 0, 7)
            assert rel_fro(k, ref[0][0][i][0]) <= TOL["bf16"] and rel_fro(v, ref[0][0][i][1]) <= TOL["bf16"]
    finally:
        s.close()
