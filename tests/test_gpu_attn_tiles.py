"""Attention tiles against the oracle at the edges of their layout: 64 query entries of one KV head, eight at a time, whose rows and
heads the query fetch deals out in two ways (up to eight heads per KV head, more), and prompts that end around a block of 64 keys.
Behind that the kernel's three uses against float64 with scores large enough to show what flat ones hide: the queries' low parts and the
softmax's moves to a new reference."""
import math

import pytest
import torch

pytestmark = pytest.mark.gpu

BASE = dict(n_layers=2, d_model=512, d_ff=1088, vocab=1024, decode_steps=2, tree_depth=3, tree_topk=3, tree_beam=3, tree_max_nodes=12)


# the tolerances are the harness's: a misplaced row would miss by the size of the values (a misplaced low part would not: see sharp_rows)
@pytest.mark.parametrize("hd,H,hkv", [(64, 8, 8), (64, 16, 4), (64, 16, 1), (64, 32, 1), (128, 8, 4), (128, 16, 2), (128, 16, 1), (64, 64, 1), (256, 4, 2), (256, 16, 1)])
@pytest.mark.parametrize("n", [3, 65])
def test_heads_per_kv_head(hd, H, hkv, n):
    _run(hd, H, hkv, n, 1)


@pytest.mark.parametrize("hd", [64, 128, 256])
@pytest.mark.parametrize("n", [63, 64, 127, 128, 129, 193])
def test_prompt_ends_around_a_key_block(hd, n):
    _run(hd, 4, 4, n, 1)


# three sequences: their rows start off the eights and tiles of the query buffer
@pytest.mark.parametrize("hd,H,hkv", [(64, 8, 8), (128, 8, 4), (256, 16, 1)])
def test_sequences_off_the_tiles(hd, H, hkv):
    _run(hd, H, hkv, 70, 3)


def _run(hd, H, hkv, n, batch):
    from tests.parity import Pair
    v = max(1, n // 2)
    pr = Pair("smolvlm2b", max_batch=batch, n_heads=H, n_kv_heads=hkv, head_dim=hd, n_visual=v, k_visual=max(1, v // 2), n_prompt=n - v, **BASE)
    try:
        for s in range(batch):
            pr.prefill(seq=s, seq_seed=s, vis_start=(n - v) // 2)
        pr.step(seqs=tuple(range(batch)))
        pr.step(seqs=tuple(reversed(range(batch))))
    finally:
        pr.close()


SIGMA = 15.0             # standard deviation of the scores (natural units)
RESCALE = 8.0            # a row's reference moves when its maximum has outgrown it by this power of two


def _rotate(x, pos, theta):
    hd = x.shape[-1]
    ang = pos.double()[:, None] * (theta ** (-2.0 * torch.arange(hd // 2, device=x.device).double() / hd))[None, :]
    c, s = ang.cos()[:, None, :], ang.sin()[:, None, :]
    a, b = x[..., :hd // 2], x[..., hd // 2:]
    return torch.cat([a * c - b * s, b * c + a * s], -1)


def _attend(q, K, V, mask, G):
    """float64 attention [rows][H * hd] and the scores [H][rows][keys]."""
    K, V = K.repeat_interleave(G, 1), V.repeat_interleave(G, 1)
    s = (torch.einsum("rhd,khd->hrk", q, K) / math.sqrt(q.shape[-1])).masked_fill(~mask, -math.inf)
    return torch.einsum("hrk,khd->rhd", torch.softmax(s, -1), V).flatten(1), s


def sharp_rows(hd, H, hkv, n, mode):
    """One launch of the attention with scores of standard deviation SIGMA, on its own: one layer, values of unit scale, the output projection an
    identity and nothing behind it, so that a row's hidden state is its input plus its attention.  Keys and values are
    the ones that the library stored.  Returns relative L2 errors against float64: the GPU's, that of queries rounded to
    bf16 (what the low parts are there to avoid), and the most often that a row's reference moves in a CTA's walk: over all keys (prompt), over a chunk of
two blocks or more (the others: 16 chunks at most)."""
    from paper_2505_19201_b200 import api, configs, synth
    dev, d, G, D, K = "cuda:0", H * hd, H // hkv, 2, 8
    v = n // 2
    p = dict(configs.PRESETS["llava7b"], n_layers=1, d_model=d, d_ff=64, vocab=512, n_heads=H, n_kv_heads=hkv, head_dim=hd, n_visual=v, k_visual=v,
             n_prompt=n - v, tree_depth=D, tree_topk=K, tree_beam=K, tree_max_nodes=K + K * K, decode_steps=4, batch=1, tap_mode=configs.TAP_FIXED, tap_layer=1)
    tw, dw = synth.target_weights(p, 5, dev), synth.draft_weights(p, 5, dev)
    eye = torch.eye(d, dtype=torch.bfloat16, device=dev)
    for w, o in ((tw["wqkv"][0], tw["wo"][0]), (dw["wqkv"], dw["wo"])):
        w[:H * hd + hkv * hd] *= math.sqrt(SIGMA / d) / 0.02
        w[H * hd + hkv * hd:] *= math.sqrt(1.0 / d) / 0.02
        o.copy_(eye)
    tw["wd"][0].zero_()
    dw["wd"].zero_()
    dw["xo"].zero_()
    ctx = api.Context(api.make_config(p), tw, dw, dev)
    try:
        vis, ids = synth.request_inputs(p, 3, dev)
        tok = torch.zeros(1, dtype=torch.int32, device=dev)
        ctx.dream_prefill(0, vis, 0, ids, tok)
        embed = lambda t: tw["embed"][torch.as_tensor(t, device=dev).long()].double()
        read = lambda what, rows, shape: torch.stack([ctx.dream_debug_read(0, what, 0, int(i)) for i in rows]).to(dev).double().view(len(rows), *shape)
        if mode == "prompt":
            rows = torch.arange(max(0, min(n, 256) - 72), min(n, 256))              # the hidden rows that can be read: of the first 256
            x, pos, w = torch.cat([vis.double(), embed(ids)])[rows.to(dev)], rows, tw["wqkv"][0]
            Kc, Vc = read(0, range(n), (hkv, hd)), read(1, range(n), (hkv, hd))
            mask = torch.arange(n)[None, :] <= rows[:, None]
        else:
            ctx.dream_compress_visual(0, v)
            tree = ctx.new_tree()
            ctx.dream_draft_tree([0], [tree])
            if mode == "verify":
                T = ctx.T
                t = tree.to_host()
                ctx.dream_verify_tree([0], [tree], torch.zeros(T, dtype=torch.int32, device=dev))
                rows, x, pos, w = torch.arange(T), embed(t["tokens"]), n + torch.tensor(t["depth"]), tw["wqkv"][0]
                Kc, Vc = read(0, range(n + T), (hkv, hd)), read(1, range(n + T), (hkv, hd))
                tail = torch.tensor([[j in t["mask"][i] for j in range(T)] for i in range(T)])
            else:
                # the second pass: the root's K best children, by score, at the tree region's rows behind the root's
                t = tree.to_host()
                level = sorted((i for i in range(ctx.T) if t["depth"][i] == 1), key=lambda i: -t["cum"][i])
                assert len(level) == K
                rows, x, pos, w = torch.arange(K), embed([t["tokens"][i] for i in level]), torch.full((K,), n + 1), dw["wqkv"]
                Kc, Vc = read(4, range(n + 1 + K), (hkv, hd)), read(5, range(n + 1 + K), (hkv, hd))
                tail = torch.cat([torch.ones(K, 1), torch.eye(K)], 1).bool()
            mask = torch.cat([torch.ones(len(rows), n, dtype=torch.bool), tail], 1)
        hidden = torch.stack([ctx.dream_debug_read(0, 7, 0, int(i)) for i in rows]).to(dev).double()
        ctx.dream_poll()
    finally:
        ctx.close()
    mask = mask.to(dev)
    norm = x / torch.sqrt((x * x).mean(-1, keepdim=True) + p["rms_eps"])
    q = _rotate((norm @ w[:H * hd].double().t()).view(len(rows), H, hd), pos.to(dev), p["rope_theta"])
    want, s = _attend(q, Kc, Vc, mask, G)
    high, _ = _attend(q.bfloat16().double(), Kc, Vc, mask, G)
    rel = lambda a: float((a - want).norm() / want.norm())
    moves = torch.zeros(s.shape[:2], device=dev)
    ref = torch.full(s.shape[:2], -math.inf, device=dev, dtype=torch.float64)
    for j in range(0, s.shape[2], 64):
        if mode != "prompt" and j % 128 == 0:
            ref.fill_(-math.inf)
        top = s[:, :, j:j + 64].amax(-1) / math.log(2.0)
        grow = (top > ref + RESCALE) & (ref > -math.inf)
        moves += grow
        ref = torch.where(grow | (ref == -math.inf), top, ref)
    return rel(hidden - x), rel(high), int(moves.max())


# A query's two parts hold 16 bits where its high part alone holds 8: the low part takes the rounding error from 2^-9 to 2^-17 of the value, by 2^8.  What
# else enters is of that size: the projection's inputs in two parts, the probabilities in two parts, fp32 sums.  Four such shares
# in all give 2^-6 of the error that the high parts alone would make; a low part with the wrong entry, twice that error.
@pytest.mark.parametrize("mode,n", [("prompt", 65), ("prompt", 250), ("prompt", 1290), ("verify", 250), ("verify", 1290), ("draft", 250), ("draft", 1290)])
@pytest.mark.parametrize("hd,H,hkv", [(64, 8, 8), (64, 64, 1), (128, 8, 4), (128, 16, 1), (256, 4, 4), (256, 16, 1)])
def test_sharp_scores(hd, H, hkv, mode, n):
    got, high, moves = sharp_rows(hd, H, hkv, n, mode)
    assert moves >= 1 or n == 65 or (n == 250 and mode != "prompt"), "the scores are too flat for what this test is about"
    assert got <= high * 2.0 ** -6, f"relative L2 error {got:.2e}, with the high parts alone {high:.2e}"
