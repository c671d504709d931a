"""Host logic of edgefm_prefill's contraction planner (tile shape and K split), checked without a GPU: invariants the kernels
rely on and its choices for the benchmark shapes."""
import itertools

from edgefm_synth import CONFIGS
from paper_2604_27476_b200 import edgefm_debug_prefill_plan

QKV, RESID, SWIGLU, QKV64 = 0, 1, 2, 3
COLUMNS = (128, 256, 64)          # output columns of the tiles the planner reports


def shapes(cfg):
    qd = cfg.n_q_heads * cfg.head_dim
    return {"qkv": (QKV if cfg.head_dim == 128 else QKV64, (cfg.n_q_heads + 2 * cfg.n_kv_heads) * cfg.head_dim, cfg.hidden), "o": (RESID, cfg.hidden, qd),
            "gate_up": (SWIGLU, cfg.ffn, cfg.hidden), "down": (RESID, cfg.hidden, cfg.ffn)}


def test_planner_invariants():
    for name, T, sms in itertools.product(CONFIGS, (1, 7, 128, 129, 511, 1023, 2047), (148, 132, 16)):
        for op, (epi, N, K) in shapes(CONFIGS[name]).items():
            tile, splits = edgefm_debug_prefill_plan(epi, T, N, K, sms)
            assert tile in (0, 1, 2) and 1 <= splits <= (8 if T <= 128 else 4)
            if epi != RESID:
                assert splits == 1, (name, op)                      # only `resid += acc` can take partial sums
            half = ((N + 63) // 64) * ((T + 127) // 128) * splits <= sms        # tiles of 64 columns fit the SMs in one round
            if epi == SWIGLU:
                assert tile == (0 if half else 1), (name, T)        # gate and up columns share one accumulator: 64 + 64 or 128 + 128
            else:
                assert (tile == 2) == (half and epi != QKV), (name, op, T)      # (a QKV tile is whole heads)
            if splits > 1:
                kb = (K + 63) // 64
                tiles = ((N + COLUMNS[tile] - 1) // COLUMNS[tile]) * ((T + 127) // 128)
                assert kb // splits >= 12                           # a unit keeps a main loop worth its fill and epilogue
                assert tiles <= sms                                 # only grids that leave SMs idle are split


def test_planner_choices_for_the_1_5b_shape():
    cfg = CONFIGS["qwen2.5-1.5b"]
    s = shapes(cfg)
    assert edgefm_debug_prefill_plan(*[s["down"][0], 2047, *s["down"][1:]], 148) == (1, 3)     # 96 wide tiles -> 288 units
    assert edgefm_debug_prefill_plan(*[s["qkv"][0], 2047, *s["qkv"][1:]], 148) == (1, 1)       # 128 wide tiles, one round
    wide, splits = edgefm_debug_prefill_plan(*[s["down"][0], 511, *s["down"][1:]], 148)
    assert splits > 1                                                                          # 48 narrow tiles alone would idle 100 SMs
    assert edgefm_debug_prefill_plan(*[s["o"][0], 511, *s["o"][1:]], 148)[1] in (1, 2)         # 24 k-blocks: at most two units


def test_planner_choices_for_a_short_prompt():
    """77 tokens of the 0.5B shape: every contraction runs with tiles of half the columns, on twice the CTAs."""
    s = shapes(CONFIGS["qwen2.5-0.5b"])
    tile = {op: edgefm_debug_prefill_plan(epi, 77, N, K)[0] for op, (epi, N, K) in s.items()}
    assert tile == {"qkv": 2, "o": 2, "gate_up": 0, "down": 2}
