"""A timeline's buffer is free when dream_trace returns, whatever other contexts of the process have under way."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def test_stop_waits_for_other_streams():
    from paper_2505_19201_b200 import api, configs, synth
    dev = "cuda:0"
    p = dict(configs.PRESETS["toy"])
    tw, dw = synth.target_weights(p, 0, dev), synth.draft_weights(p, 0, dev)
    vis, ids = synth.request_inputs(p, 0, dev)
    other = torch.cuda.Stream()
    traced, busy = api.Context(api.make_config(p), tw, dw, dev), api.Context(api.make_config(p), tw, dw, dev, stream=other)
    try:
        torch.cuda.synchronize()
        for stop in (True, False):                       # stopped, or given another buffer
            traced.dream_trace(1000)
            first = traced._trace
            with torch.cuda.stream(other):
                torch.cuda._sleep(100_000_000)           # some 50 ms: the kernels behind it are queued long before they run
                busy.dream_seq_reset(0)
                busy.dream_prefill(0, vis, 0, ids)
                done = torch.cuda.Event()
                done.record(other)
            if stop:
                traced.dream_trace(0)
            else:
                traced.dream_trace(1000)
            assert done.query(), "kernels of another context may still hold the buffer"
            traced.dream_trace(0)
            n = int(first[0])
            torch.cuda.synchronize()
            assert int(first[0]) == n
        busy.dream_poll()
    finally:
        traced.close()
        busy.close()
