"""Top-k and log-sum-exp at block edges, with ties, signed zeros and infinities, against a stable sort in float64.
Values and ids are exact.  Log-sum-exp: the exponentials are good to some 2^-21 and their sums, over a thread's columns, a block and the
blocks, to 30 roundings or so, each 2^-24 of a sum that is at least 1; with the rounding of a result below 32 (2^-20) less than 2e-5."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def run(x, k):
    from paper_2505_19201_b200 import api
    rows = x.shape[0]
    tv, ti, ls = (torch.zeros(rows, k, device="cuda"), torch.zeros(rows, k, dtype=torch.int32, device="cuda"), torch.zeros(rows, device="cuda"))
    api.dream_topk_lse_static(x, k, tv, ti, ls)
    torch.cuda.synchronize()
    order = torch.sort(x.double().cpu(), dim=1, descending=True, stable=True)
    assert torch.equal(ti.cpu().long(), order.indices[:, :k])
    assert torch.equal(tv.cpu().double() + 0.0, order.values[:, :k] + 0.0)
    ref = torch.logsumexp(x.double().cpu(), 1)
    assert float((ls.cpu().double() - ref).abs().max()) < 2e-5


@pytest.mark.parametrize("V", [16, 1000, 1023, 4096, 4097, 8192, 32001, 262144])
@pytest.mark.parametrize("rows,k", [(1, 1), (3, 2), (61, 2), (10, 10), (8, 16)])
def test_random(V, rows, k):
    g = torch.Generator(device="cuda").manual_seed(V + rows)
    run(torch.randn(rows, V, device="cuda", generator=g) * 3, k)


@pytest.mark.parametrize("V", [64, 4100, 12288])
def test_ties_zeros_infinities(V):
    g = torch.Generator(device="cuda").manual_seed(V)
    x = torch.randint(-2, 3, (7, V), device="cuda", generator=g).float()      # many ties: the lower id wins
    x[1] = 0.0
    x[1, ::3] = -0.0
    x[2] = -5.0
    x[3, :] = -float("inf")
    x[3, 5] = -1.0
    x[3, V - 1] = -1.0
    x[3, V // 2] = -2.0
    run(x[:3].contiguous(), 16)
    run(x[3:4].contiguous(), 3)


# The same through a context, whose draft passes and small verifications take blocks of 1024 columns (each of its columns in a
# thread's four): rows and list lengths on either side of the choice, widths around a block's end
@pytest.mark.parametrize("V", [16, 1000, 1022, 1023, 1024, 1025, 4096, 4100, 8193, 65536])
@pytest.mark.parametrize("rows,k", [(1, 1), (1, 16), (7, 10), (18, 16), (19, 2), (256, 2)])
def test_context_blocks(V, rows, k):
    from paper_2505_19201_b200 import api, configs, synth
    p = configs.scaled("toy", vocab=V, decode_steps=2)
    ctx = api.Context(api.make_config(p), synth.target_weights(p, 0, "cuda:0"), synth.draft_weights(p, 0, "cuda:0"), "cuda:0")
    try:
        g = torch.Generator(device="cuda").manual_seed(V + rows)
        for x in (torch.randn(rows, V, device="cuda", generator=g) * 3, torch.randint(-2, 3, (rows, V), device="cuda", generator=g).float() * 0.5 - 0.0):
            tv, ti, ls = (torch.zeros(rows, k, device="cuda"), torch.zeros(rows, k, dtype=torch.int32, device="cuda"), torch.zeros(rows, device="cuda"))
            ctx.dream_debug_topk(x, k, tv, ti, ls)
            ctx.dream_poll()
            order = torch.sort(x.double().cpu(), dim=1, descending=True, stable=True)
            assert torch.equal(ti.cpu().long(), order.indices[:, :k])
            assert torch.equal(tv.cpu().double() + 0.0, order.values[:, :k] + 0.0)
            assert float((ls.cpu().double() - torch.logsumexp(x.double().cpu(), 1)).abs().max()) < 2e-5
    finally:
        ctx.close()
