"""The bounded waits of the barrier-free step kernel, through the library's self-test kernel: the two words behind the status word
hold what each of them did."""
import pytest

import workloads as wl
from parity_util import make_session

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def outcomes():
    """The status block's first words, and how long the self-test kernel took (seconds)."""
    import torch

    import paper_2410_08391_b200 as kvp
    pair = wl.PairCfg("t", wl.uniform_model(1, 64, 2, 1, 64, 128, 97), wl.uniform_model(1, 64, 2, 1, 64, 128, 97), (0,))
    s = make_session(pair, wl.make_weights(pair, seed=1), wl.custom_prompts(97, [8], seed=1))
    try:
        s.workspace[:256].zero_()
        torch.cuda.synchronize()
        kvp.kvp_selftest_wait_timeout(s.h, s.workspace, s.stream)      # (the first launch loads the kernel)
        torch.cuda.synchronize()
        s.workspace[:256].zero_()
        torch.cuda.synchronize()
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record(s.torch_stream)
        kvp.kvp_selftest_wait_timeout(s.h, s.workspace, s.stream)
        b.record(s.torch_stream)
        torch.cuda.synchronize()
        return s.workspace[:16].view(torch.int32).cpu().tolist(), a.elapsed_time(b) * 1e-3
    finally:
        s.close()


def test_every_kind_of_wait_runs_out(outcomes):
    assert outcomes[0][:3] == [1, 1, 1]      # DEV_TIMEOUT from the mbarrier wait, the tagged value, the sleeping loader


def test_limits_are_a_few_seconds(outcomes):
    """The kernel waits with a 64th of the limits, which are meant to be two seconds: at most five with room for a slower clock."""
    assert 0.005 < outcomes[1] < 5.0 / 64
