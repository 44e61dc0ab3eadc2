"""The tensor-core GEMM at the edges of its tiles and forms, against a float64 matmul.

Tolerance: activations enter as a high and a low bf16 part (what is dropped is below 2^-17 of each), the
partial products are exact in fp32 and a sum of K terms is rounded at most once per MMA, so the error stays
below (2^-17 + K / 16 * 2^-24) * sum_k |x_k w_k|."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2505_19201_b200 import api, configs, synth
    p = configs.scaled("llava7b", n_layers=1, vocab=1024, n_visual=64, k_visual=16, n_prompt=32, decode_steps=2)
    tw, dw = synth.target_weights(p, 0, "cuda:0"), synth.draft_weights(p, 0, "cuda:0")
    c = api.Context(api.make_config(p), tw, dw, "cuda:0")
    yield c
    c.close()


def check(ctx, rows, N, K, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    W = (torch.randn(N, K, device="cuda", generator=g) * 0.02).to(torch.bfloat16)
    X = torch.randn(rows, K, device="cuda", generator=g)
    out = ctx.dream_debug_gemm(W, X, 1)
    ctx.dream_poll()
    ref = X.double() @ W.double().t()
    bound = (2.0 ** -17 + K / 16 * 2.0 ** -24) * (X.double().abs() @ W.double().abs().t()) + 1e-12
    assert bool(((out.double() - ref).abs() <= bound).all()), f"rows {rows} N {N} K {K}"


# both planes in one MMA: 1..128 rows, one, two or four accumulators, one or two panels per stage;
# two MMAs: 129..256 rows
@pytest.mark.parametrize("rows", [1, 7, 8, 9, 16, 17, 31, 32, 33, 63, 64, 65, 72, 73, 96, 127, 128, 129, 144, 145, 176, 255, 256])
def test_rows(ctx, rows):
    check(ctx, rows, 776, 704, rows)


# k panels per accumulator: one short of, equal to and one past a chain; a tile shared by several pairs
@pytest.mark.parametrize("K", [64, 128, 448, 512, 576, 1024, 1088, 4096])
@pytest.mark.parametrize("rows", [24, 200])
def test_panels(ctx, rows, K):
    check(ctx, rows, 520, K, K + rows)


# output columns: less than one CTA's half, ragged halves, more tiles than pairs
@pytest.mark.parametrize("N", [8, 120, 128, 136, 248, 256, 264, 22016])
@pytest.mark.parametrize("rows", [61, 244])
def test_columns(ctx, rows, N):
    check(ctx, rows, N, 320, N + rows)


# shares of whole pairs per tile: two per tile exactly and not quite, as long as allowed and one unit longer, a last
# share shorter than the others, more pairs per tile than panels
@pytest.mark.parametrize("N,K", [(9472, 576), (9728, 576), (8192, 3840), (4096, 11008), (6144, 5120), (2048, 2048), (256, 128)])
@pytest.mark.parametrize("rows", [9, 61, 244])
def test_shares(ctx, rows, N, K):
    check(ctx, rows, N, K, N + K)


# three pairs per two tiles: an even and an odd number of tiles, the most and the fewest, too few panels for it
@pytest.mark.parametrize("N,K", [(12288, 4096), (12032, 4096), (12544, 576), (9728, 320), (12800, 576), (12288, 256), (12288, 128)])
@pytest.mark.parametrize("rows", [9, 61, 244])
def test_three_pairs(ctx, rows, N, K):
    check(ctx, rows, N, K, N + K)
