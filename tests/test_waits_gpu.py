"""The bounded waits of the barrier-free step kernel, through the library's self-test kernel: words 1 to 3 behind the status word
hold what each of them did."""
import pytest

import workloads as wl
from parity_util import make_session

pytestmark = pytest.mark.gpu


def _outcomes():
    import torch

    import paper_2410_08391_b200 as kvp
    pair = wl.PairCfg("t", wl.uniform_model(1, 64, 2, 1, 64, 128, 97), wl.uniform_model(1, 64, 2, 1, 64, 128, 97), (0,))
    s = make_session(pair, wl.make_weights(pair, seed=1), wl.custom_prompts(97, [8], seed=1))
    try:
        s.workspace[:256].zero_()
        torch.cuda.synchronize()
        kvp.kvp_selftest_wait_timeout(s.h, s.workspace, s.stream)
        torch.cuda.synchronize()
        return s.workspace[:16].view(torch.int32).cpu().tolist()
    finally:
        s.close()


def test_loader_stops_when_its_consumers_gave_up():
    words = _outcomes()
    assert words[0] == 1      # the wait that nobody satisfies ran out (DEV_TIMEOUT)
    assert words[3] == 1      # a free slot is not filled any more once the consumers have given up
