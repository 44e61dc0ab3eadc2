"""Attention tiles against the oracle at the edges of their layout: 64 query entries of one KV head, eight at a time, whose rows and
heads the query fetch deals out in two ways (up to eight heads per KV head, more), and prompts that end around a block of 64 keys."""
import pytest

pytestmark = pytest.mark.gpu

BASE = dict(n_layers=2, d_model=512, d_ff=1088, vocab=1024, decode_steps=2, tree_depth=3, tree_topk=3, tree_beam=3, tree_max_nodes=12)


# the tolerances are the harness's: the layout changes no rounding, a misplaced row would miss by the size of the values
@pytest.mark.parametrize("hd,H,hkv", [(64, 8, 8), (64, 16, 4), (64, 16, 1), (64, 32, 1), (128, 8, 4), (128, 16, 2), (128, 16, 1), (256, 4, 2), (256, 16, 1)])
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
