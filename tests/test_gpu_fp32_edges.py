"""The fp32 GEMM and attention at the edges of their tiles: GEMM against a float64 matmul (fp32 sums of K terms:
error below K * 2^-24 * sum_k |x_k w_k|), attention through whole rounds against the oracle at key counts around
the number of warps and of keys in flight."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2505_19201_b200 import api, configs, synth
    p = dict(configs.PRESETS["toy"])
    tw, dw = synth.target_weights(p, 0, "cuda:0"), synth.draft_weights(p, 0, "cuda:0")
    c = api.Context(api.make_config(p), tw, dw, "cuda:0")
    yield c
    c.close()


@pytest.mark.parametrize("rows", [1, 4, 5, 8, 9, 15, 256])
@pytest.mark.parametrize("N,K,shift", [(256, 256, 0), (1, 1, 0), (3, 7, 0), (33, 128, 0), (30, 129, 0), (17, 260, 1), (257, 1000, 0), (64, 1024, 1), (2048, 512, 0)])
def test_gemm(ctx, rows, N, K, shift):
    g = torch.Generator(device="cuda").manual_seed(rows * 7 + N + K)
    W = torch.randn(N * K + 4, device="cuda", generator=g)[shift:shift + N * K].view(N, K)      # shift 1: not 16-byte aligned
    X = torch.randn(rows, K, device="cuda", generator=g)
    out = ctx.dream_debug_gemm(W, X)
    ctx.dream_poll()
    ref = X.double() @ W.double().t()
    assert bool(((out.double() - ref).abs() <= K * 2.0 ** -24 * (X.double().abs() @ W.double().abs().t()) + 1e-12).all())


@pytest.mark.parametrize("n_visual,n_prompt", [(1, 1), (4, 3), (6, 2), (7, 2), (20, 11), (24, 9)])
@pytest.mark.parametrize("track_entropy", [0, 1])
def test_rounds(n_visual, n_prompt, track_entropy):
    from tests.parity import Pair
    pr = Pair("toy", n_visual=n_visual, k_visual=(n_visual + 1) // 2, n_prompt=n_prompt, decode_steps=4, track_entropy=track_entropy)
    try:
        pr.prefill()
        for _ in range(2):
            pr.step()
    finally:
        pr.close()
