"""What the prompt's contractions are launched as (host logic, no GPU): invariants the kernels rely on, over the benchmark shapes and odd ones."""
import itertools

from edgefm_synth import CONFIGS
from paper_2604_27476_b200 import edgefm_debug_prefill_launch, edgefm_debug_prefill_plan
from test_prefill_plan import QKV, RESID, SWIGLU, shapes

ODD = {"odd": (RESID, 1000, 72), "one_column_tile": (RESID, 8, 8), "wide_ffn": (SWIGLU, 18952, 264), "heads": (QKV, 384, 4104)}


def tiles(M, N, columns):
    return -(-M // 128) * -(-N // columns)


def test_launches():
    ops = [op for name in CONFIGS for op in shapes(CONFIGS[name]).values()] + list(ODD.values())
    for (epi, N, K), M, sms in itertools.product(ops, (1, 8, 15, 64, 77, 121, 128, 129, 256, 257, 384, 1000, 2048, 4096), (148, 132, 20)):
        columns, splits, cluster, pairs, swapped = edgefm_debug_prefill_launch(epi, M, N, K, sms)
        step, kb = (columns // 2 if epi == SWIGLU else columns), -(-K // 64)
        what = (epi, M, N, K, sms)
        assert columns % 16 == 0 and 64 <= columns <= 256, what
        if cluster:
            assert splits == 1 and not pairs and columns in (64, 128, 256), what
            assert 1 <= cluster <= min(8, kb), what                           # no CTA without a k-block
            assert tiles(min(M, 128) if swapped else M, N, step) * cluster <= sms or (epi == SWIGLU and M <= 128 and cluster == 1 and tiles(M, N, step) <= 2 * sms), what   # one or two CTAs per SM
        else:
            assert columns in (128, 256) or (pairs and epi == RESID), what
            assert 1 <= splits <= 8 and (splits == 1 or epi == RESID), what
        if pairs:
            assert M > 128 and columns > 128, what                            # tiles of 128 columns are launched as single CTAs'
        if swapped:                    # fewer padded tokens than columns, both pieces side by side; or two row tiles that share weight tiles
            assert cluster and columns <= 128 and (-(-M // 8) * 8 < columns if M < 128 else 128 < M <= 256), what
        if epi == QKV:
            assert columns % 128 == 0, what                                   # whole heads of 128
        if epi == SWIGLU:
            assert columns in (128, 256), what


def test_clusters_run_at_once():
    """A partial tile of more than half an SM's shared memory (256 columns; 217 and more swapped rows) leaves one CTA per SM, and of such clusters
    only so many fit the GPCs: one tile more is a second round (0.5B shape, 450 tokens: 20 clusters of seven where 15 run at once)."""
    one_per_sm = (0, 148, 74, 45, 33, 26, 22, 15, 15)
    for name, M in itertools.product(CONFIGS, itertools.chain(range(8, 700, 8), range(700, 4097, 100))):
        for op, (epi, N, K) in shapes(CONFIGS[name]).items():
            columns, _, cluster, _, swapped = edgefm_debug_prefill_launch(epi, M, N, K)
            rows = M if swapped and M > 128 else min(M, 128)
            if cluster and rows * columns * 4 > 109 * 1024:
                assert tiles(min(M, 128) if swapped else M, N, columns // 2 if epi == SWIGLU else columns) <= one_per_sm[cluster], (name, op, M)


def test_short_prompts_share_the_k_of_a_tile():
    """77 tokens of the 0.5B shape: QKV, O and down run on 98 to 126 CTAs instead of 14 to 18."""
    s = shapes(CONFIGS["qwen2.5-0.5b"])
    for op, least in (("qkv", 5), ("o", 7), ("down", 8)):
        epi, N, K = s[op]
        assert edgefm_debug_prefill_launch(epi, 77, N, K)[2] >= least, op


def test_columns_fill_the_rounds_of_the_7b_shape():
    """4096 tokens: tiles of 256 columns would take four rounds for 3.03 rounds of work."""
    epi, N, K = shapes(CONFIGS["qwen2.5-7b-32k"])["down"]
    columns, splits, cluster, pairs, _ = edgefm_debug_prefill_launch(epi, 4096, N, K)
    assert (splits, cluster, pairs) == (1, 0, 1)
    units = 16 * -(-N // columns)
    assert units / (-(-units // 74) * 74) > 0.95
    assert edgefm_debug_prefill_plan(epi, 4096, N, K) == (1, 1)
