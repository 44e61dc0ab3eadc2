"""A device-side wait that nothing ends becomes an error: the CTA that waited gives up at its limit, its partner at once with
it, dream_poll names the wait, and the context's kernels still run."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("limit_ms", [1, 50])
def test_expired_wait(limit_ms):
    from paper_2505_19201_b200 import api, configs, synth
    p = configs.scaled("toy", decode_steps=2)
    dev = "cuda:0"
    tw, dw = synth.target_weights(p, 0, dev), synth.draft_weights(p, 0, dev)
    ctx = api.Context(api.make_config(p), tw, dw, dev)
    sec = torch.full((2,), -1.0, device=dev)
    ctx.dream_debug_wait(limit_ms, sec)
    t0 = time.monotonic()
    with pytest.raises(api.DreamError) as e:
        ctx.dream_poll()
    assert e.value.code == -6 and "k_wait_probe" in str(e.value)
    assert time.monotonic() - t0 < 2.0
    first, second = sec.tolist()
    # an attempt may overstay by its own suspension, a millisecond, and either CTA starts a little after the other
    assert limit_ms * 1e-3 <= first < limit_ms * 1e-3 + 0.05 and 0 < second < limit_ms * 1e-3 + 0.1
    vis, ids = synth.request_inputs(p, 0, dev)
    first_token = torch.full((1,), -1, dtype=torch.int32, device=dev)
    ctx.dream_prefill(0, vis, 0, ids, first_token)
    torch.cuda.synchronize()
    assert 0 <= int(first_token) < p["vocab"]
    for bad in (0, 1001):
        with pytest.raises(api.DreamError) as e:
            ctx.dream_debug_wait(bad, sec)
        assert e.value.code == -1
    ctx.close()
