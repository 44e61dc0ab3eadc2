"""The GEMM forms of a prompt (several token tiles, full waves of tiles, epilogues that gate or rotate) against float64.

Tolerance of a sum as in test_gpu_gemm_edges: (2^-17 + K / 16 * 2^-24) * sum_k |x_k w_k|, for the dropped part of the activations
and one rounding per MMA.  What an epilogue adds is stated where it is checked."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def context(model, v, q, **over):
    from paper_2505_19201_b200 import api, configs, synth
    p = configs.scaled(model, n_layers=1, vocab=1024, n_visual=v, k_visual=16, n_prompt=q, decode_steps=2, **over)
    tw, dw = synth.target_weights(p, 0, DEV), synth.draft_weights(p, 0, DEV)
    return p, tw, api.Context(api.make_config(p), tw, dw, DEV)


@pytest.fixture(scope="module")
def ctx():
    p, tw, c = context("llava7b", 640, 640)
    yield c
    c.close()


def operands(rows, N, K):
    g = torch.Generator(device=DEV).manual_seed(rows + N + K)
    return (torch.randn(N, K, device=DEV, generator=g) * 0.02).to(torch.bfloat16), torch.randn(rows, K, device=DEV, generator=g)


def sums(W, X, K):
    """The float64 products and the bound of the kernel's error."""
    return X.double() @ W.double().t(), (2.0 ** -17 + K / 16 * 2.0 ** -24) * (X.double().abs() @ W.double().abs().t()) + 1e-12


# tiles (256 columns x a token tile) on 74 pairs: exactly a wave (N 9472 at two token tiles), a rest so small that a wave is given
# up (9728 at two, 7680 at five), an ordinary rest, fewer tiles than pairs, a ragged last tile, one panel
@pytest.mark.parametrize("N,K", [(9472, 576), (9728, 576), (7680, 1024), (12288, 4096), (4096, 704), (9480, 320), (264, 64)])
@pytest.mark.parametrize("rows", [257, 512, 513, 832, 1279, 1280])
def test_store(ctx, rows, N, K):
    W, X = operands(rows, N, K)
    out = ctx.dream_debug_gemm(W, X, 1)
    ctx.dream_poll()
    ref, bound = sums(W, X, K)
    assert bool(((out.double() - ref).abs() <= bound).all())


# 256 rows take the row kernel, 257 the epilogue; widths: full waves and a rest, no full wave, a last tile of half a width
@pytest.mark.parametrize("ff,K", [(11008, 4096), (4736, 576), (1088, 576), (64, 64)])
@pytest.mark.parametrize("rows", [9, 256, 257, 513, 832, 1280])
def test_gate(ctx, rows, ff, K):
    W, X = operands(rows, 2 * ff, K)
    out = ctx.dream_debug_gemm(W, X, 2)
    ctx.dream_poll()
    ref, bound = sums(W, X, K)
    g, u, eg, eu = ref[:, :ff], ref[:, ff:], bound[:, :ff], bound[:, ff:]
    act = g * torch.sigmoid(g) * u
    # |silu'| <= 1.1; __expf is off by up to 2 + 1.16 |g| ulp, division and products by a few; the result is kept as two bf16 parts (2^-17)
    tol = 1.1 * eg * (u.abs() + eu) + torch.sigmoid(g) * g.abs() * eu + act.abs() * (2.0 ** -17 + (8 + 2 * g.abs()) * 2.0 ** -24) + 1e-12
    assert bool(((out.double() - act).abs() <= tol).all())


# rotary and the append to the pages: the cache rows of the first layer are rotations of projected, normalised embeddings
@pytest.mark.parametrize("model,v,q", [("smolvlm2b", 300, 213), ("llava7b", 832, 447), ("llava13b", 100, 157), ("pixtral12b", 512, 1), ("gemma3_12b", 700, 580)])
def test_rotary_and_append(model, v, q):
    from paper_2505_19201_b200 import synth
    p, tw, c = context(model, v, q)
    try:
        vis, ids = synth.request_inputs(p, 0, DEV)
        at = q // 2
        c.dream_prefill(0, vis, at, ids)
        c.dream_poll()
        n, H, Hkv, hd, d = v + q, p["n_heads"], p["n_kv_heads"], p["head_dim"], p["d_model"]
        emb = tw["embed"][ids.long()]
        x = torch.cat([emb[:at], vis, emb[at:]]).double()
        x = x / torch.sqrt((x * x).mean(1, keepdim=True) + p["rms_eps"]) * tw["ln1"][0].double()
        half = torch.arange(hd // 2, dtype=torch.float64, device=DEV)
        for r in sorted({0, 1, 127, 128, 143, 144, 255, 256, 257, n // 2, n - 2, n - 1} & set(range(n))):
            ref, bound = sums(tw["wqkv"][0][H * hd:], x[r:r + 1], d)
            k, vv = ref[0, :Hkv * hd].view(Hkv, hd), ref[0, Hkv * hd:]
            ang = r * p["rope_theta"] ** (-2.0 * half / hd)
            cos, sin = torch.cos(ang), torch.sin(ang)
            a, b = k[:, :hd // 2], k[:, hd // 2:]
            k = torch.cat([a * cos - b * sin, b * cos + a * sin], 1).flatten()
            err = 2 * float(bound.max()) + 3e-6 * float(ref.abs().max())           # a rotation mixes two sums; fp32 norm, sine and cosine
            for what, want in ((0, k), (1, vv)):
                got = c.dream_debug_read(0, what, 0, r).double().to(DEV)
                assert bool(((got - want).abs() <= want.abs() * 2.0 ** -8 + err).all()), (model, r, what)      # the cache is bf16
    finally:
        c.close()


# the tensor core truncates when it accumulates: a chain of n MMAs loses half an ulp of its running sum, on average half the
# chain's, per MMA, n * 2^-25 of a sum of one sign; chains are KB / 8 panels of eight MMAs, four to eight
@pytest.mark.parametrize("K", [512, 2048, 3840, 4096])
@pytest.mark.parametrize("rows", [129, 256, 257, 1280])
def test_bias_of_same_sign_sums(ctx, rows, K):
    W, X = operands(rows, 2048, K)
    W, X = W.abs(), X.abs()
    out = ctx.dream_debug_gemm(W, X, 1)
    ctx.dream_poll()
    ref = X.double() @ W.double().t()
    assert abs(float(((out.double() - ref) / ref).mean())) <= 8 * min(8, max(4, K // 64 // 8)) * 2.0 ** -25
