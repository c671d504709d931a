"""The decode-step kernel where its cuts change: every way a row can be cut (whole in tiles of 16 or of 8 rows, segments as
tensor-map boxes or row by row), activations whole or by segments, tiles against head halves and batches, builds for 1, 2, 4
and 8 tokens, both cache formats -- each against the oracle's plain decode steps of the same tokens."""
import numpy as np
import pytest

from edgefm_synth import CONFIGS, first_token
from helpers import Pair, TOKEN_MARGIN, assert_logits_close, top2_margin

pytestmark = pytest.mark.gpu

BASE = CONFIGS["tiny"].with_(n_layers=2, vocab=300, n_q_heads=4, n_kv_heads=2, head_dim=64, hidden=256, ffn=512)
# name: (shape, cached positions, tokens per call, cache format).  148 CTAs: rows per CTA are the operator's rows / 148, rounded up.
CASES = {
    # 16 whole rows fit up to 2176 columns, 8 up to 4096; 2200 and 2248 are no multiples of 64 (a last block is padded)
    "whole_16_last": (dict(hidden=2176), 20, 1, None),
    "whole_8_first_ragged": (dict(hidden=2200), 20, 1, None),
    "whole_8_first_ragged_4": (dict(hidden=2200), 20, 4, None),
    "whole_8_last": (dict(hidden=4096, ffn=1400), 20, 1, None),
    "whole_8_two_sets": (dict(hidden=2248, ffn=1400), 20, 8, None),
    "boxes": (dict(hidden=4160, ffn=1400), 20, 1, None),
    "boxes_2": (dict(hidden=4160, n_q_heads=8, n_kv_heads=1), 20, 2, None),
    "boxes_8": (dict(hidden=4160, ffn=1400), 20, 8, None),
    "row_segments": (dict(hidden=4168), 20, 1, None),
    "row_segments_4": (dict(hidden=4168), 20, 4, None),
    # the down projection's long rows: 25 rows per CTA as 13 + 12, activations by segments; 6 and 17 rows
    "down_boxes_13": (dict(hidden=3584, ffn=18944, n_layers=1), 20, 1, None),
    "down_boxes_13_2": (dict(hidden=3584, ffn=18944, n_layers=1), 20, 2, None),
    "down_row_segments": (dict(hidden=2504, ffn=11208, n_layers=1), 20, 1, None),
    "down_segments_4": (dict(hidden=888, ffn=6104, n_layers=1), 20, 4, None),
    # more units per CTA than a batch of partial sums holds: heads 37 pairs (cut at halves of 64), vocabulary 700 rows
    "batches_1": (dict(n_q_heads=40, n_kv_heads=8, head_dim=128, vocab=103000, n_layers=1), 20, 1, None),
    "batches_8": (dict(n_q_heads=72, n_kv_heads=9, head_dim=128, vocab=7000, n_layers=1), 20, 8, None),
    # fewer rows than CTAs
    "narrow": (dict(hidden=72, ffn=40, n_q_heads=1, n_kv_heads=1), 3, 1, None),
    "narrow_8": (dict(hidden=72, ffn=40, n_q_heads=1, n_kv_heads=1), 3, 8, None),
    # more attention outputs than 128 per CTA: few rows (and so few CTAs) with many heads; 24576 on all CTAs (tables out of shared memory)
    "few_rows_many_heads": (dict(hidden=8, n_q_heads=44, n_kv_heads=22, head_dim=128, ffn=40), 20, 1, None),
    "few_rows_many_heads_int8": (dict(hidden=8, n_q_heads=44, n_kv_heads=22, head_dim=128, ffn=40), 20, 1, "int8"),
    "few_rows_many_heads_2": (dict(hidden=8, n_q_heads=15, n_kv_heads=3, head_dim=128, ffn=64), 20, 2, None),
    "few_rows_many_heads_4": (dict(hidden=8, n_q_heads=12, n_kv_heads=3, head_dim=128, ffn=256), 20, 4, None),
    "few_rows_many_heads_8": (dict(hidden=8, n_q_heads=12, n_kv_heads=3, head_dim=128, ffn=256), 20, 8, None),
    "outputs_24576": (dict(hidden=152, n_q_heads=192, n_kv_heads=24, head_dim=128, n_layers=1), 20, 1, None),
    # vectors that leave no room for tables and chunk lists, then for smaller chunks only, then for half blocks of cached positions, too
    "far_tables": (dict(hidden=24056, n_kv_heads=4, ffn=160, n_layers=1), 300, 1, None),
    "small_chunks_boxes": (dict(hidden=28800, n_kv_heads=4, ffn=64, n_layers=1), 300, 1, None),
    "small_chunks_rows": (dict(hidden=30600, n_kv_heads=4, ffn=64, n_layers=1), 300, 1, "int8"),
    "half_blocks_rows_2": (dict(hidden=15600, n_q_heads=8, n_kv_heads=4, ffn=64, n_layers=1), 148 * 8 + 21, 2, None),
    "half_blocks_boxes_2": (dict(hidden=15616, n_q_heads=8, n_kv_heads=4, head_dim=128, ffn=64, n_layers=1), 148 * 8 + 21, 2, None),
    "small_chunks_4": (dict(hidden=11000, n_q_heads=8, n_kv_heads=4, ffn=64, n_layers=1), 40, 4, None),
    # attention: tiles of 16 positions in quarters, blocks of 64 (heads of 128) or 128; one position, one more than a tile, than a block
    **{f"attention_{d}_{n}_{m}{q or ''}": (dict(head_dim=d, n_q_heads=g, n_kv_heads=1), n, m, q)
       for d, g in ((64, 3), (128, 8)) for n, m, q in ((1, 1, None), (17, 2, None), (148 * 16 + 1, 1, None), (148 * 64 + 5, 1, None), (148 * 128 + 9, 8, None),
                                                        (1, 1, "int8"), (33, 8, "int8"), (148 * 64 + 5, 1, "int8"), (148 * 128 + 9, 1, "int8"))},
}


@pytest.mark.parametrize("name", list(CASES))
def test_cuts_match_the_oracle(name):
    import torch
    more, T0, m, kv = CASES[name]
    cfg = BASE.with_(**more)
    rounds = 3
    pair = Pair(cfg, seed=len(name), cache_len=T0, max_context=T0 + rounds * m + 1, kv_format=kv, block_tokens=m if m in (2, 4) else 0)
    try:
        tok, pos = first_token(cfg) % cfg.vocab, T0
        for r in range(rounds):
            if m == 1:
                ref, nxt = pair.oracle.step(tok, pos)
                pair.ctx.step(tok, pos)
                torch.cuda.synchronize()
                pair.ctx.sync_status()
                got, refs = [pair.ctx.logits.cpu().numpy()], [ref]
                acc = 1
            else:
                n0, t, p, block = pair.oracle.cur_len, tok, pos, [tok]
                for _ in range(m - 1):                       # proposals: the oracle's own continuation, wrong from a place on
                    _, t = pair.oracle.step(t, p)
                    p += 1
                    block.append(t)
                pair.oracle.truncate(n0)
                if r != 1:
                    block[m // 2] = (block[m // 2] + 1) % cfg.vocab
                refs, acc, nxt = pair.oracle.verify_block(block, pos)
                pair.ctx.verify_block(block, pos)
                torch.cuda.synchronize()
                pair.ctx.sync_status()
                got = pair.ctx.block_logits.cpu().numpy()
            for t in range(acc):
                assert_logits_close(got[t], refs[t], f"{name} round {r} token {t}")
            if any(top2_margin(refs[t]) <= TOKEN_MARGIN for t in range(acc)):
                break                                        # a near-tie: the two sides may continue with different tokens
            if m > 1:
                assert int(pair.ctx.n_accepted.item()) == acc
            assert int(pair.ctx.next_token.item()) == nxt
            if m > 1:
                assert pair.ctx.sync_length() == pair.oracle.cur_len
            tok, pos = nxt, pos + acc
    finally:
        pair.close()
