"""Rows of the residual stream at the edges of the norm's split into blocks of 2048 columns, few rows (a decode round)
and many (a prompt pass of more than 256), up to the widest model; the oracle's bounds."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", [960, 1024, 1088, 2048, 2112, 5120, 16384])
@pytest.mark.parametrize("preset,n_prompt", [("toy", 16), ("smolvlm2b", 16), ("smolvlm2b", 240)])
def test_row_widths(preset, n_prompt, d):
    from tests.parity import Pair
    pr = Pair(preset, n_visual=24, k_visual=8, n_prompt=n_prompt, n_layers=2, d_model=d, n_heads=4, n_kv_heads=2, head_dim=64, d_ff=256, vocab=512,
              decode_steps=2, tree_depth=2, tree_topk=2, tree_beam=2, tree_max_nodes=7)
    try:
        pr.prefill()
        pr.step()
    finally:
        pr.close()
