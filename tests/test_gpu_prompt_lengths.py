"""Prompts whose rows end just before, at and behind the edges of a token tile (256), of a pass over the prompt
(1280) and of the row counts at which the projections change form, on a small bf16 model against the oracle."""
import pytest

pytestmark = pytest.mark.gpu

SMALL = dict(n_layers=2, d_model=512, n_heads=8, n_kv_heads=4, head_dim=64, d_ff=1088, vocab=1024, decode_steps=2, tree_depth=3, tree_topk=3,
             tree_beam=3, tree_max_nodes=12)


@pytest.mark.parametrize("n", [2, 64, 128, 129, 256, 257, 300, 513, 769, 1279, 1281, 2561])
@pytest.mark.parametrize("draft_blocks", [1, 3])
def test_prompt(n, draft_blocks):
    from tests.parity import Pair
    v = max(1, n // 2 + 1)
    pr = Pair("smolvlm2b", n_visual=v, k_visual=max(1, v // 2), n_prompt=n - v, draft_blocks=draft_blocks, **SMALL)
    try:
        pr.prefill(vis_start=(n - v) // 3)
        pr.step()
    finally:
        pr.close()


def test_wide_model_long_prompt():
    """As many token tiles as give full waves of tiles and a stream-K rest, at a real model's widths."""
    from tests.parity import Pair
    pr = Pair("llava7b", n_layers=1, n_visual=700, k_visual=100, n_prompt=620, decode_steps=2, tap_lo=1, tap_hi=1)
    try:
        pr.prefill()
        pr.step()
    finally:
        pr.close()
