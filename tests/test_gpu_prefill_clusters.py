"""Prompt kernels whose work is shared out inside clusters, at the sizes where a share is empty or ragged: contractions whose K tiles are
fewer than a cluster's CTAs or whose rows are, key blocks fewer than the CTAs of a query tile (early query tiles then leave some without any),
pairs of row tiles with an odd one left over.  Tolerances: those of the prompt's other parity tests (two-piece operands, fp32 sums)."""
import pytest

from edgefm_synth import CONFIGS
from test_gpu_prefill import run_case

pytestmark = pytest.mark.gpu

BASE = CONFIGS["tiny"].with_(qkv_bias=True)
CASES = {
    # contractions by clusters: (shape changes, cached positions, tokens)
    "one_k_tile": (dict(hidden=64, n_q_heads=1, n_kv_heads=1, ffn=72, vocab=40), 0, 17),
    "k_tiles_less_than_a_cluster": (dict(hidden=200, ffn=328), 2, 9),
    "rows_less_than_a_cluster": (dict(hidden=1024, ffn=4096, n_layers=1, vocab=300), 0, 8),
    "ragged_row_groups": (dict(hidden=1024, ffn=4096, n_layers=1, vocab=300), 0, 27),
    "row_tile_less_one": (dict(hidden=264, ffn=2056), 0, 127),
    "three_row_tiles_one_row": (dict(hidden=264, ffn=520), 0, 257),
    "odd_head_in_a_tile_of_two": (dict(n_q_heads=5, n_kv_heads=1, ffn=200), 0, 140),
    "heads_of_128_by_clusters": (dict(hidden=1152, n_q_heads=6, n_kv_heads=2, head_dim=128, ffn=1032, n_layers=1, vocab=300), 40, 61),
    # two row tiles as the columns of one row of tiles: one token into the second, a ragged group of 16, all of it, one token too many
    "two_row_tiles_first": (dict(hidden=1024, ffn=4096, n_layers=1, vocab=300), 0, 129),
    "two_row_tiles_ragged": (dict(hidden=1152, n_q_heads=6, n_kv_heads=2, head_dim=128, ffn=1032, n_layers=1, vocab=300), 5, 201),
    "two_row_tiles_full": (dict(hidden=264, ffn=520), 0, 256),
    "two_row_tiles_one_k_tile": (dict(hidden=64, n_q_heads=1, n_kv_heads=1, ffn=72, vocab=40), 0, 250),
    # the persistent kernel, row tiles in pairs: an even number, an odd one, a last tile of one row
    "pairs_even": (dict(ffn=9480, n_layers=1, vocab=500), 0, 256),
    "pairs_odd": (dict(ffn=9480, n_layers=1, vocab=500), 3, 300),
    "pairs_last_row": (dict(ffn=9480, n_layers=1, vocab=500), 0, 385),
    # attention by clusters
    "blocks_less_than_ctas": (dict(n_layers=1, vocab=500), 150, 20),
    "early_tiles_without_blocks": (dict(n_layers=1, vocab=500), 0, 500),
    "many_blocks": (dict(n_layers=1, vocab=500), 2100, 130),
    "many_blocks_heads_of_128": (dict(n_layers=1, vocab=500, n_q_heads=2, n_kv_heads=1, head_dim=128), 1500, 33),
    "one_block_each": (dict(n_layers=1, vocab=500), 1000, 24),
}


@pytest.mark.parametrize("name", list(CASES))
def test_shares_of_a_cluster_match_the_oracle(name):
    more, T0, n = CASES[name]
    run_case(BASE.with_(**more), T0, n, 700 + len(name))
