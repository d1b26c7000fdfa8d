"""Two host threads, each with a handle of its own, on one stream: launches of one kernel with different amounts of shared memory
must not disturb one another (the limit of dynamic shared memory is an attribute of the kernel, not of the launch)."""
import threading

import numpy as np
import pytest

import workloads as wl
from parity_util import make_session

pytestmark = pytest.mark.gpu


def _pairs(dtype):
    if dtype == "bf16":      # 1 and 4 query heads per kv head: same kernel, other scratch
        return [wl.PairCfg("g%d" % g, wl.uniform_model(1, 64, 2, 1, 64, 128, 211), wl.uniform_model(1, 128, 2 * g, 2, 64, 128, 211), (0,)) for g in (1, 4)]
    return [wl.PairCfg("f%d" % f, wl.uniform_model(1, 64, 2, 1, 16, 96, 211), wl.uniform_model(1, 64, 2, 2, 16, f, 211), (0,), dtype="f32") for f in (96, 8192)]


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_two_threads_with_different_models(dtype):
    import torch
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):      # both sessions take it: their kernels follow one another
        sessions, results, errors = [], [None, None], []
        for pair in _pairs(dtype):
            pr = wl.custom_prompts(211, [40], seed=2)
            s = make_session(pair, wl.make_weights(pair, seed=2, regime="fanin"), pr, extra_len=2)
            s.prefill_predict(torch.from_numpy(pr.tokens).to(s.device), [40])
            s.poll()
            sessions.append(s)
        tok = torch.tensor([7], dtype=torch.int32, device="cuda")
    want = []
    for s in sessions:
        with torch.cuda.stream(stream):
            s.cache.seq_lens.fill_(40)
            logits, _ = s.decode_step(tok, [40])
            s.poll()
            want.append(logits.cpu().numpy())
    go = threading.Barrier(2)

    def work(i):
        try:
            s = sessions[i]
            torch.cuda.set_device(0)
            with torch.cuda.stream(stream):
                go.wait()
                for _ in range(500):
                    s.cache.seq_lens.fill_(40)
                    logits, _ = s.decode_step(tok, [40])
                s.poll()
                results[i] = logits.cpu().numpy()
        except Exception as e:      # noqa: BLE001  (told to the test's own thread)
            errors.append(e)

    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for got, ref in zip(results, want):
        assert np.allclose(got, ref, rtol=1e-5, atol=1e-5)
    for s in sessions:
        s.close()
