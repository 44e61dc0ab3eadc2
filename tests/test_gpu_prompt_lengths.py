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


# as many token tiles as give full waves of tiles (whose projections finish in the GEMM's epilogue) and a stream-K
# rest, at real models' widths: head_dim 128 in two passes, 64, 128 with grouped queries, 256; an odd gate width
@pytest.mark.parametrize("model,over", [
    ("llava7b", dict(n_visual=700, k_visual=100, n_prompt=620)),
    ("smolvlm2b", dict(n_visual=900, k_visual=100, n_prompt=252)),
    ("smolvlm2b", dict(n_visual=300, k_visual=100, n_prompt=701, d_ff=8000)),
    ("pixtral12b", dict(n_visual=500, k_visual=100, n_prompt=250)),
    ("gemma3_12b", dict(n_visual=256, k_visual=64, n_prompt=901)),
])
def test_wide_models(model, over):
    from tests.parity import Pair
    pr = Pair(model, n_layers=1, vocab=2048, decode_steps=2, tap_lo=1, tap_hi=1, **over)
    try:
        pr.prefill(vis_start=over["n_prompt"] // 2)
        pr.step()
    finally:
        pr.close()
