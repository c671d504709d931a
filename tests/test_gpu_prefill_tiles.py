"""Prompt contractions at the sizes where the tile shape changes: half-width tiles are taken where they fit the SMs in one round
(148 of them: 9472 columns for up to 128 tokens, 4736 for up to 256), with ragged last tiles, one and two row tiles, heads of 64 (half-width
QKV tiles) and of 128 (whole ones), and an output matrix whose rows are no multiple of the four a warp takes at a time."""
import pytest

from edgefm_synth import CONFIGS
from test_gpu_prefill import run_case

pytestmark = pytest.mark.gpu

BASE = CONFIGS["tiny"].with_(qkv_bias=True)
CASES = {
    "ragged_columns": (dict(hidden=264, ffn=72, vocab=301), 20, 77),
    "one_tile": (dict(hidden=64, n_q_heads=1, n_kv_heads=1, ffn=64, vocab=37), 0, 8),
    "row_tile_full": (dict(hidden=264, ffn=200), 3, 128),
    "row_tile_full_plus_one": (dict(hidden=264, ffn=200), 3, 129),
    "gate_up_last_half_width": (dict(ffn=9472, n_layers=1, vocab=500), 0, 40),
    "gate_up_first_full_width": (dict(ffn=9480, n_layers=1, vocab=500), 0, 40),
    "two_row_tiles_last_half_width": (dict(ffn=4736, n_layers=1, vocab=500), 0, 140),
    "two_row_tiles_first_full_width": (dict(ffn=4744, n_layers=1, vocab=500), 0, 140),
    "heads_of_128": (dict(hidden=328, n_q_heads=3, n_kv_heads=1, head_dim=128, ffn=136), 50, 65),
}


@pytest.mark.parametrize("name", list(CASES))
def test_tile_shapes_match_the_oracle(name):
    more, T0, n = CASES[name]
    run_case(BASE.with_(**more), T0, n, 500 + len(name))
