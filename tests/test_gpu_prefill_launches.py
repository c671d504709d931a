"""The persistent contraction kernel of long prompts, in every form the planner launches: QKV, O / down and gate/up by single CTAs of 128 and 256 columns and
by pairs of CTAs with an even and an odd number of row tiles, every width that pairs take (multiples of 16, most of them with a last chunk
that reaches past the tile and a ragged last tile), with K splits and the norm behind them, K longer and shorter than the ring.  Norm weights are
random and there are two layers, so that the scales, weights and cache rows that one contraction leaves for the next are seen.  Every case
states the plan it is there for.  Tolerances: those of the prompt's other parity tests (two-piece operands, fp32 sums)."""
import pytest

from edgefm_synth import CONFIGS, make_weights
from helpers import random_norms
from test_gpu_prefill import run_case
from test_gpu_prefill_clusters import check_plan

pytestmark = pytest.mark.gpu

BASE = CONFIGS["tiny"].with_(qkv_bias=True, vocab=300)


def shape(hidden, n_q_heads, n_kv_heads, head_dim, ffn):
    return dict(hidden=hidden, n_q_heads=n_q_heads, n_kv_heads=n_kv_heads, head_dim=head_dim, ffn=ffn)


def pairs(columns):
    """O and down in pairs of CTAs, tiles of that many columns."""
    return {"o": (columns, 1, 0, 1, 0), "down": (columns, 1, 0, 1, 0)}


SINGLE_128, SINGLE_256, PAIRS_256 = (128, 1, 0, 0, 0), (256, 1, 0, 0, 0), (256, 1, 0, 1, 0)
#: (shape, cached positions, tokens, what runs: operator -> (columns, splits, cluster, pairs, swapped))
CASES = {
    "qkv_single_128": (shape(64, 16, 2, 128, 1648), 0, 1817, {"qkv": SINGLE_128, "gate_up": PAIRS_256}),
    "qkv_single_256": (shape(64, 14, 2, 64, 128), 0, 3585, {"qkv": SINGLE_256}),
    "qkv_pairs": (shape(328, 16, 2, 128, 64), 3, 904, {"qkv": PAIRS_256}),
    "qkv_pairs_odd": (shape(64, 14, 2, 128, 64), 0, 1080, {"qkv": PAIRS_256}),
    "gate_up_single": (shape(328, 1, 1, 64, 4864), 0, 258, {"gate_up": SINGLE_256}),
    "gate_up_pairs": (shape(328, 1, 1, 128, 9568), 0, 133, {"gate_up": PAIRS_256}),
    "gate_up_pairs_odd": (shape(328, 4, 2, 64, 3144), 7, 273, {"gate_up": PAIRS_256}),
    "added_single_128": (shape(3672, 1, 1, 64, 64), 0, 1178, {"o": SINGLE_128, "down": SINGLE_128}),
    "added_single_256": (shape(3200, 1, 1, 64, 328), 0, 1310, {"o": SINGLE_256, "down": SINGLE_256}),
    "down_single_split": (shape(3776, 5, 1, 64, 5736), 0, 8, {"down": (256, 7, 0, 0, 0)}),
    "o_single_split": (shape(3200, 12, 2, 128, 128), 0, 609, {"o": (256, 2, 0, 0, 0)}),
    "o_pairs_split": (shape(2704, 12, 2, 128, 64), 0, 397, {"o": (256, 2, 0, 1, 0)}),
    "o_pairs_split_odd": (shape(3584, 12, 2, 128, 64), 0, 261, {"o": (256, 2, 0, 1, 0)}),
    "pairs_144": (shape(3176, 1, 1, 64, 64), 0, 653, pairs(144)),
    "pairs_144_odd": (shape(1728, 1, 1, 64, 128), 0, 1343, pairs(144)),
    "pairs_160": (shape(3584, 1, 1, 64, 64), 0, 658, pairs(160)),
    "pairs_160_odd": (shape(2784, 1, 1, 64, 64), 0, 784, pairs(160)),
    "pairs_176": (shape(3072, 1, 1, 64, 64), 0, 908, pairs(176)),
    "pairs_176_odd": (shape(3072, 1, 1, 64, 328), 5, 782, pairs(176)),
    "pairs_192": (shape(3200, 1, 1, 64, 64), 0, 923, pairs(192)),
    "pairs_192_odd": (shape(3200, 1, 1, 64, 64), 0, 774, pairs(192)),
    "pairs_208": (shape(3584, 1, 1, 64, 64), 0, 901, pairs(208)),
    "pairs_208_odd": (shape(3592, 1, 1, 64, 64), 0, 771, pairs(208)),
    "pairs_224": (shape(3064, 1, 1, 64, 64), 0, 1156, pairs(224)),
    "pairs_224_odd": (shape(3832, 1, 1, 64, 64), 0, 789, pairs(224)),
    "pairs_240": (shape(3200, 1, 1, 64, 64), 0, 1203, pairs(240)),
    "pairs_240_odd": (shape(3200, 1, 1, 64, 64), 0, 1070, pairs(240)),
    "pairs_256": (shape(3384, 1, 1, 64, 328), 0, 1166, pairs(256)),
    "pairs_256_odd": (shape(3584, 1, 1, 64, 64), 0, 1037, pairs(256)),
    "pairs_last_row": (shape(3072, 1, 1, 64, 64), 0, 769, pairs(176)),
    "tiles_of_256_in_clusters": (shape(856, 4, 2, 128, 64), 0, 265, {"qkv": (256, 1, 7, 0, 0), "o": (256, 1, 8, 0, 0)}),
}


@pytest.mark.parametrize("name", list(CASES))
def test_contractions_of_long_prompts_match_the_oracle(name):
    more, T0, n, expected = CASES[name]
    cfg = BASE.with_(**more)
    check_plan(cfg, T0, n, expected)
    run_case(cfg, T0, n, 900 + len(name), weights=random_norms(make_weights(cfg), len(name)))
