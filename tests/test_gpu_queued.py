"""Calls made while earlier work of the stream is still pending: a host that runs requests ahead of the GPU gets the
results of the same calls made one at a time.

The stream is held by a sleeping kernel, so that everything the calls read back or copy (the snapshots of the verified
lengths, the page lists) is still outstanding when the next call is made."""
import pytest
import torch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"
HOLD = 600_000_000            # clocks, a third of a second: the calls below are enqueued in a few milliseconds


def model():
    from paper_2505_19201_b200 import configs, synth
    p = configs.scaled("smolvlm2b", n_layers=2, d_model=512, n_heads=8, n_kv_heads=4, d_ff=1024, vocab=1024, n_visual=40, k_visual=10, n_prompt=30,
                       tree_depth=2, tree_topk=2, tree_beam=2, tree_max_nodes=6, batch=2, decode_steps=8)
    return p, synth.target_weights(p, 0, DEV), synth.draft_weights(p, 0, DEV)


def context(p, tw, dw):
    from paper_2505_19201_b200 import api
    return api.Context(api.make_config(p, max_batch=2, page_tokens=16), tw, dw, DEV)


def round_of(ctx, p, seqs):
    """One round; the verified logits and the accepted lengths."""
    T, n = ctx.T, len(seqs)
    trees = [ctx.new_tree() for _ in seqs]
    am, acc = torch.zeros(n * T, dtype=torch.int32, device=DEV), torch.zeros(n, dtype=torch.int32, device=DEV)
    tok = torch.zeros(n * (p["tree_depth"] + 1), dtype=torch.int32, device=DEV)
    lg = torch.zeros(n * T, p["vocab"], device=DEV)
    ctx.dream_draft_tree(seqs, trees)
    ctx.dream_verify_tree(seqs, trees, am, None, lg)
    ctx.dream_accept(seqs, trees, am, acc, tok)
    return [lg, acc, tok]


def start(ctx, p, seq, seed):
    from paper_2505_19201_b200 import synth
    vis, ids = synth.request_inputs(p, seed, DEV)
    ctx.dream_seq_reset(seq)
    ctx.dream_prefill(seq, vis, 5, ids)
    ctx.dream_compress_visual(seq, p["k_visual"])


def requests(ctx, p, hold):
    """Two requests in a row on sequence 0, two rounds each, then one on sequence 1."""
    if hold:
        torch.cuda._sleep(HOLD)
    out = []
    for seq, seed in ((0, 0), (0, 1), (1, 2)):
        start(ctx, p, seq, seed)
        out += round_of(ctx, p, [seq]) + round_of(ctx, p, [seq])
    return out


def test_requests_ahead_of_the_gpu():
    p, tw, dw = model()
    ctx = context(p, tw, dw)
    ref = [t.cpu() for t in requests(ctx, p, False)]
    ctx.dream_poll()
    out = requests(ctx, p, True)
    other = context(p, tw, dw)                  # a context made meanwhile
    ctx.dream_poll()
    other.dream_poll()
    assert all(torch.equal(a, b.cpu()) for a, b in zip(ref, out))
    other.close()
    ctx.close()


def swapped(ctx, p, hold):
    """Both sequences decode a round; then sequence 0 starts anew on the pages that sequence 1 gave back."""
    if hold:
        torch.cuda._sleep(HOLD)
    start(ctx, p, 0, 0)
    start(ctx, p, 1, 1)
    out = round_of(ctx, p, [0, 1])
    ctx.dream_seq_reset(0)
    ctx.dream_seq_reset(1)
    start(ctx, p, 0, 2)
    return out + round_of(ctx, p, [0])


def test_pages_change_hands_ahead_of_the_gpu():
    p, tw, dw = model()
    res = []
    for hold in (False, True):
        ctx = context(p, tw, dw)
        ctx.dream_poll()
        res.append([t.cpu() for t in swapped(ctx, p, hold)])
        ctx.dream_poll()
        ctx.close()
    assert all(torch.equal(a, b) for a, b in zip(*res))
