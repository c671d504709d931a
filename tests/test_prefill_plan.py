"""Host logic of edgefm_prefill's contraction planner (output tiles and K units, as edgefm_debug_prefill_plan reports them), checked without a
GPU: that the query says what runs, invariants the kernels rely on, and its choices for the benchmark shapes."""
import itertools

from edgefm_synth import CONFIGS
from paper_2604_27476_b200 import edgefm_debug_prefill_launch, edgefm_debug_prefill_plan

QKV, RESID, SWIGLU, QKV64 = 0, 1, 2, 3
COLUMNS = (128, 256, 64)          # output columns of the tiles the query reports (1: at most)


def shapes(cfg):
    qd = cfg.n_q_heads * cfg.head_dim
    return {"qkv": (QKV if cfg.head_dim == 128 else QKV64, (cfg.n_q_heads + 2 * cfg.n_kv_heads) * cfg.head_dim, cfg.hidden), "o": (RESID, cfg.hidden, qd),
            "gate_up": (SWIGLU, cfg.ffn, cfg.hidden), "down": (RESID, cfg.hidden, cfg.ffn)}


def test_planner_invariants():
    for name, T, sms in itertools.product(CONFIGS, (1, 7, 128, 129, 511, 1023, 2047), (148, 132, 16)):
        for op, (epi, N, K) in shapes(CONFIGS[name]).items():
            tile, units = edgefm_debug_prefill_plan(epi, T, N, K, sms)
            columns, splits, cluster, _, _ = edgefm_debug_prefill_launch(epi, T, N, K, sms)
            what = (name, op, T, sms)
            assert tile == {64: 2, 128: 0}.get(columns, 1) and units == max(splits, cluster), what      # the query says what runs
            assert 1 <= splits <= (8 if T <= 128 else 4), what
            half = ((N + 63) // 64) * ((T + 127) // 128) <= sms                  # tiles of 64 columns fit the SMs in one round
            if epi == SWIGLU:
                assert tile in (0, 1), what                                      # gate and up columns share one accumulator: 64 + 64 or 128 + 128
                assert tile == 0 or not half, what
            elif tile == 2:
                assert half and epi != QKV, what                                 # (a QKV tile is whole heads)
            if epi != RESID:
                assert splits == 1, what                                         # only `resid += acc` can take partial sums
            if splits > 1:
                kb = (K + 63) // 64
                tiles = ((N + COLUMNS[tile] - 1) // COLUMNS[tile]) * ((T + 127) // 128)
                assert kb // splits >= 12, what                                  # a unit keeps a main loop worth its fill and epilogue
                assert tiles <= sms, what                                        # only grids that leave SMs idle are split


def test_planner_choices_for_the_1_5b_shape():
    cfg = CONFIGS["qwen2.5-1.5b"]
    s = shapes(cfg)
    assert edgefm_debug_prefill_launch(*[s["down"][0], 2047, *s["down"][1:]]) == (176, 1, 0, 1, 0)   # 72 tiles on 74 pairs of SMs, no partial sums
    assert edgefm_debug_prefill_plan(*[s["down"][0], 2047, *s["down"][1:]], 148) == (1, 1)
    assert edgefm_debug_prefill_plan(*[s["qkv"][0], 2047, *s["qkv"][1:]], 148) == (1, 1)       # 64 pairs of wide tiles, one round
    for op in ("o", "down"):
        assert edgefm_debug_prefill_plan(*[s[op][0], 511, *s[op][1:]], 148)[1] > 1             # 24 tiles of 256 columns alone would idle most SMs


def test_planner_choices_for_a_short_prompt():
    """77 tokens of the 0.5B shape: every contraction runs with tiles of half the columns, on twice the CTAs."""
    s = shapes(CONFIGS["qwen2.5-0.5b"])
    tile = {op: edgefm_debug_prefill_plan(epi, 77, N, K)[0] for op, (epi, N, K) in s.items()}
    assert tile == {"qkv": 2, "o": 2, "gate_up": 0, "down": 2}
