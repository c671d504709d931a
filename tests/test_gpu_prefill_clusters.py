"""Prompt kernels whose work is shared out, at the sizes where a share is empty or ragged: contractions whose K tiles are fewer than a cluster's
CTAs or whose rows are, two row tiles as the columns of one row of tiles, pairs of row tiles with an odd one left over, attention whose key
blocks are dealt to several CTAs of which those of early query tiles may get none.  Every case states the plan it is there for.  Tolerances:
those of the prompt's other parity tests (two-piece operands, fp32 sums)."""
import pytest

from edgefm_synth import CONFIGS, make_weights
from helpers import random_norms
from test_gpu_prefill import run_case
from test_prefill_plan import shapes

pytestmark = pytest.mark.gpu

BASE = CONFIGS["tiny"].with_(qkv_bias=True)
SMALL = dict(n_layers=1, vocab=500)
#: (shape changes, cached positions, tokens, what runs: operator -> (columns, splits, cluster, pairs, swapped); "parts" -> CTAs per query tile)
CASES = {
    # contractions by clusters
    "one_k_tile": (dict(hidden=64, n_q_heads=1, n_kv_heads=1, ffn=72, vocab=40), 0, 17, {"qkv": (64, 1, 1, 0, 1), "down": (64, 1, 1, 0, 1)}),
    "six_k_tiles_one_cta": (dict(hidden=200, ffn=328), 2, 9, {"down": (64, 1, 1, 0, 1)}),
    "rows_one_per_cta": (dict(hidden=1024, ffn=4096, n_layers=1, vocab=300), 0, 8, {"down": (64, 1, 8, 0, 1)}),
    "ragged_row_groups": (dict(hidden=1024, ffn=4096, n_layers=1, vocab=300), 0, 27, {"down": (64, 1, 8, 0, 1)}),
    "row_tile_less_one": (dict(hidden=264, ffn=2056), 0, 127, {"qkv": (64, 1, 5, 0, 0), "gate_up": (128, 1, 3, 0, 0), "down": (64, 1, 7, 0, 0)}),
    "three_row_tiles_one_row": (dict(hidden=264, ffn=520), 0, 257, {"qkv": (64, 1, 5, 0, 0), "gate_up": (128, 1, 5, 0, 0)}),
    "odd_head_in_a_tile_of_two": (dict(n_q_heads=5, n_kv_heads=1, ffn=200), 0, 140, {"qkv": (64, 1, 1, 0, 0), "o": (64, 1, 5, 0, 0)}),
    "heads_of_128_by_clusters": (dict(hidden=1152, n_q_heads=6, n_kv_heads=2, head_dim=128, ffn=1032, n_layers=1, vocab=300), 40, 61, {"qkv": (128, 1, 6, 0, 1)}),
    # two row tiles as the columns of one row of tiles: one token into the second, a ragged group of 16, all of it (the partial tile, 128 KB, is larger
    # than the ring), all of it in one k-block
    "two_row_tiles_first": (dict(hidden=1808, n_q_heads=4, n_kv_heads=2, head_dim=128, ffn=632, vocab=300), 0, 129,
                            {op: (128, 1, c, 0, 1) for op, c in (("qkv", 8), ("o", 8), ("gate_up", 8), ("down", 5))}),
    "two_row_tiles_ragged": (dict(hidden=1152, n_q_heads=6, n_kv_heads=2, head_dim=128, ffn=1032, n_layers=1, vocab=300), 5, 201, {"gate_up": (128, 1, 6, 0, 1)}),
    "two_row_tiles_full": (dict(hidden=264, ffn=1032), 0, 256, {"gate_up": (128, 1, 5, 0, 1)}),
    "two_row_tiles_full_added": (dict(hidden=3584, n_q_heads=1, n_kv_heads=1, ffn=4096, **SMALL), 0, 256, {"gate_up": (128, 1, 2, 0, 1), "down": (128, 1, 4, 0, 1)}),
    "two_row_tiles_one_k_tile": (dict(hidden=64, n_q_heads=1, n_kv_heads=1, ffn=8192, vocab=40), 0, 250, {"gate_up": (128, 1, 1, 0, 1)}),
    # the persistent kernel, row tiles in pairs: an even number, an odd one, an odd one of one row
    "pairs_even": (dict(ffn=9480, **SMALL), 0, 256, {"gate_up": (256, 1, 0, 1, 0)}),
    "pairs_odd": (dict(ffn=3144, **SMALL), 3, 300, {"gate_up": (256, 1, 0, 1, 0)}),
    "pairs_last_row": (dict(ffn=3144, **SMALL), 0, 257, {"gate_up": (256, 1, 0, 1, 0)}),
    # attention: shares of several sizes, and early query tiles with fewer blocks than CTAs
    "blocks_not_shared_out": (dict(**SMALL), 150, 20, {"parts": 1}),
    "two_blocks_each": (dict(**SMALL), 1000, 24, {"parts": 4}),
    "early_tiles_without_blocks": (dict(**SMALL), 0, 1000, {"parts": 4}),
    "early_tiles_without_blocks_heads_of_128": (dict(n_q_heads=2, n_kv_heads=1, head_dim=128, **SMALL), 100, 700, {"parts": 4}),
    "many_blocks": (dict(**SMALL), 2100, 130, {"parts": 9}),
    "many_blocks_heads_of_128": (dict(n_q_heads=2, n_kv_heads=1, head_dim=128, **SMALL), 1500, 33, {"parts": 6}),
}


def check_plan(cfg, T0, n, expected):
    from paper_2604_27476_b200 import edgefm_debug_prefill_attention, edgefm_debug_prefill_launch
    got = {op: edgefm_debug_prefill_launch(epi, n, N, K) for op, (epi, N, K) in shapes(cfg).items()}
    got["parts"] = edgefm_debug_prefill_attention(n, T0, cfg.n_q_heads)
    assert {op: got[op] for op in expected} == expected


@pytest.mark.parametrize("name", list(CASES))
def test_shares_of_a_cluster_match_the_oracle(name):
    more, T0, n, expected = CASES[name]
    cfg = BASE.with_(**more)
    check_plan(cfg, T0, n, expected)
    run_case(cfg, T0, n, 700 + len(name), weights=random_norms(make_weights(cfg)))
