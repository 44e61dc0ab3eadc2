"""Whole calls at odd sizes of the real model widths: every call returns, the status word stays clear, what comes out is finite,
and the first round of a second request with the same prompt repeats the first one's bits."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def tree_parents(T, depth, topk):
    """Breadth first, topk children a node, no deeper than `depth`."""
    parent, dep = [-1], [0]
    for i in range(T):
        if i < len(parent) and dep[i] < depth:
            for _ in range(topk):
                if len(parent) < T:
                    parent.append(i)
                    dep.append(dep[i] + 1)
    return parent


# model, layers, visual, kept, prompt, vis_start, depth, topk, nodes, batch, draft blocks, entropies, page
@pytest.mark.parametrize("model,L,v,k,q,vs,D,K,N,B,blocks,ent,page", [
    ("smolvlm2b", 3, 28, 21, 37, 0, 6, 5, 35, 1, 1, 0, 32),          # 65 prompt rows
    ("smolvlm2b", 2, 22, 5, 268, 44, 5, 10, 12, 2, 1, 1, 128),       # 290: two token tiles
    ("smolvlm2b", 2, 126, 126, 2170, 7, 4, 1, 4, 3, 3, 0, 16),       # two passes, a chain, the three-block draft over a long context
    ("llava7b", 2, 24, 24, 85, 27, 3, 1, 3, 1, 3, 1, 128),
    ("llava7b", 3, 368, 276, 687, 510, 6, 9, 37, 4, 3, 0, 64),
    ("llava7b", 2, 16, 4, 16, 16, 3, 10, 100, 2, 1, 0, 32),          # 32 prompt rows, 202 rows verified
    ("llava13b", 2, 70, 35, 294, 36, 7, 6, 64, 3, 3, 1, 128),
    ("llava13b", 2, 148, 37, 37, 0, 4, 9, 16, 4, 1, 0, 64),
    ("pixtral12b", 2, 116, 29, 1513, 1473, 5, 1, 5, 1, 3, 0, 16),
    ("pixtral12b", 2, 738, 184, 128, 0, 7, 8, 24, 3, 1, 1, 128),
    ("gemma3_12b", 2, 92, 92, 62, 0, 7, 8, 58, 3, 3, 1, 16),         # 154 rows: one tile of more than 128
    ("gemma3_12b", 2, 512, 384, 327, 14, 7, 7, 81, 1, 3, 0, 64),
])
def test_calls_return(model, L, v, k, q, vs, D, K, N, B, blocks, ent, page):
    from paper_2505_19201_b200 import api, configs, synth
    p = configs.scaled(model, n_layers=L, n_visual=v, k_visual=k, n_prompt=q, tree_depth=D, tree_topk=K, tree_beam=K, tree_max_nodes=N, batch=B,
                       draft_blocks=blocks, track_entropy=ent, vocab=8192, decode_steps=30)
    ctx = api.Context(api.make_config(p, page_tokens=page), synth.target_weights(p, 0, DEV), synth.draft_weights(p, 0, DEV), DEV)
    T, seqs, V = ctx.T, list(range(B)), p["vocab"]
    i32 = lambda n: torch.zeros(n, dtype=torch.int32, device=DEV)
    drafted, trees = [ctx.new_tree() for _ in seqs], [ctx.new_tree() for _ in seqs]
    for b, t in enumerate(trees):
        t.load([(7 * b + 13 * i) % V for i in range(T)], tree_parents(T, D, K))
    am, acc, tok, lg = i32(B * T), i32(B), i32(B * (D + 1)), torch.zeros(B * T, V, device=DEV)
    first, ae, scores = i32(B), torch.zeros(B, L, device=DEV), torch.zeros(B, v, device=DEV)
    prompts = [synth.request_inputs(p, b, DEV) for b in seqs]
    seen = []
    try:
        for _ in range(2):
            for b, (vis, ids) in enumerate(prompts):
                ctx.dream_seq_reset(b)
                ctx.dream_prefill(b, vis, vs, ids, first[b:b + 1], None, ae[b], None)
                ctx.dream_compress_visual(b, k, None, None, scores[b])
            ctx.dream_poll()
            for i in range(8):
                ctx.dream_draft_tree(seqs, drafted)
                ctx.dream_verify_tree(seqs, trees, am, None, lg)
                ctx.dream_accept(seqs, trees, am, acc, tok)
                if i == 0:
                    seen.append([t.clone() for t in (lg, am, first, ae, scores)])
            ctx.dream_poll()
            assert all(bool(torch.isfinite(t).all()) for t in (lg, ae, scores))
            assert all(bool(torch.isfinite(t.cum_logp).all()) for t in drafted)
        assert all(torch.equal(x, y) for x, y in zip(*seen))
    finally:
        ctx.close()
