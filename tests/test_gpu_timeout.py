"""The bounded device-side waits of the step kernel, driven to expiry without any fault: its exchanges are told to expect what no CTA
sends (another tag; an arrival more than there are CTAs) and the bound is shortened to 2 ms, so the first exchange of the next step
gives up.  The kernel must return, the status must read EDGEFM_ERR_TIMEOUT, the context must still be destroyable, and a
fresh context on the same weights must work."""
import time

import pytest

from edgefm_synth import CONFIGS, first_token
from helpers import Pair, assert_logits_close

pytestmark = pytest.mark.gpu


def test_exchange_wait_expires_and_is_reported():
    import torch
    from paper_2604_27476_b200 import (DecodeContext, EdgefmError, Status, edgefm_debug_set_wait_limit, edgefm_sync_status)
    cfg = CONFIGS["tiny"]
    pair = Pair(cfg, max_context=cfg.cache_len + 8)
    try:
        stream = torch.cuda.current_stream().cuda_stream
        tok, pos = first_token(cfg), cfg.first_position
        ref, nxt = pair.oracle.step(tok, pos)
        pair.ctx.step(tok, pos)                                   # a normal step first
        edgefm_sync_status(pair.ctx.handle, stream)
        assert_logits_close(pair.ctx.logits.cpu().numpy(), ref, "before")
        edgefm_debug_set_wait_limit(pair.ctx.handle, 2_000_000, 1)    # 2 ms; the exchanges now wait for what nobody sends
        t0 = time.perf_counter()
        pair.ctx.step(nxt, pos + 1)
        with pytest.raises(EdgefmError) as ei:
            edgefm_sync_status(pair.ctx.handle, stream)
        dt = time.perf_counter() - t0
        assert ei.value.status == Status.ERR_TIMEOUT
        assert dt < 2.0                                            # the kernel returned by itself, well inside a second
        with pytest.raises(EdgefmError):                           # limits are validated
            edgefm_debug_set_wait_limit(pair.ctx.handle, 10, 0)
        # the CUDA context is intact: a fresh edgefm context on the same weights computes the right answer
        other = DecodeContext(cfg, pair.ptrs, cfg.cache_len + 8)
        other.prefill_kv(pair.kd, pair.vd)
        other.step(tok, pos)
        torch.cuda.synchronize()
        assert_logits_close(other.logits.cpu().numpy(), ref, "fresh context after the expired wait")
        other.close()
    finally:
        pair.close()                                               # destroying the timed-out context succeeds


@pytest.mark.parametrize("m,block_tokens", [(1, 0), (4, 4), (8, 0)], ids=["step", "block4", "block8"])
@pytest.mark.parametrize("limit_ns", [1000, 200_000])
def test_a_cta_that_gives_up_waits_for_its_copies(m, block_tokens, limit_ns):
    """Waits so short that every CTA gives up with its copies under way (1 us: before the first chunk is there; 200 us: the whole of this
    small step has been asked for and the feeding threads are done).  The copies must land before the CTA's shared memory is
    someone else's: other contexts, whose kernels follow at once on the same stream, compute what they always do."""
    import torch
    from paper_2604_27476_b200 import DecodeContext, EdgefmError, Status, edgefm_debug_set_wait_limit
    cfg = CONFIGS["tiny"]
    pair = Pair(cfg, max_context=cfg.cache_len + 8, block_tokens=block_tokens)
    others = [DecodeContext(cfg, pair.ptrs, cfg.cache_len + 8, block_tokens=block_tokens) for _ in range(3)]
    try:
        tok, pos = first_token(cfg), cfg.first_position
        ref, _ = pair.oracle.step(tok, pos)
        block = [tok] + [5] * (m - 1)
        run = lambda ctx: ctx.step(tok, pos) if m == 1 else ctx.verify_block(block, pos)
        for o in others:
            o.prefill_kv(pair.kd, pair.vd)
        torch.cuda.synchronize()
        edgefm_debug_set_wait_limit(pair.ctx.handle, limit_ns, 1)
        run(pair.ctx)
        for o in others:
            run(o)
        torch.cuda.synchronize()
        with pytest.raises(EdgefmError) as ei:
            pair.ctx.sync_status()
        assert ei.value.status == Status.ERR_TIMEOUT
        for o in others:
            o.sync_status()
            assert_logits_close(o.logits.cpu().numpy(), ref, "a context behind the one that gave up")
    finally:
        for o in others:
            o.close()
        pair.close()


@pytest.mark.parametrize("m,block_tokens,kv_format", [(1, 0, None), (4, 4, None), (8, 0, None), (1, 0, "int8"), (8, 0, "int8")],
                         ids=["step", "block4", "block8", "step_int8", "block8_int8"])
def test_a_timeout_is_not_forgotten(m, block_tokens, kv_format):
    """Behind an expired wait the exchange buffers hold what a step left that was never finished.  Neither new cache rows nor a prompt nor
    further steps, with the bound restored, may make the context look sound again: the status stays until it is destroyed."""
    import torch
    from paper_2604_27476_b200 import EdgefmError, Status, edgefm_debug_set_wait_limit
    cfg = CONFIGS["tiny"]
    pair = Pair(cfg, cache_len=32, max_context=128, block_tokens=block_tokens, kv_format=kv_format)
    try:
        tok, pos = first_token(cfg), 32
        run = lambda: pair.ctx.step(tok, pos) if m == 1 else pair.ctx.verify_block([tok] + [5] * (m - 1), pos)

        def expired():
            with pytest.raises(EdgefmError) as ei:
                pair.ctx.sync_status()
            return ei.value.status == Status.ERR_TIMEOUT

        run()
        pair.ctx.sync_status()
        pair.ctx.append_kv(32)
        edgefm_debug_set_wait_limit(pair.ctx.handle, 2_000_000, 1)
        run()
        assert expired()
        edgefm_debug_set_wait_limit(pair.ctx.handle, 1_000_000_000, 0)
        pair.ctx.prefill_kv(pair.kd, pair.vd)
        assert expired()
        pair.ctx.append_kv(32)
        pair.ctx.next_token.fill_(-7)
        run()
        assert expired()
        assert int(pair.ctx.next_token.item()) == -7              # the step did nothing
        pair.ctx.append_kv(30)
        pair.ctx.prefill(list(range(1, 12)), 30)
        assert expired()
    finally:
        torch.cuda.synchronize()
        pair.close()


def test_prefill_contraction_wait_expires_and_is_reported():
    """The same for the contractions of edgefm_prefill: their stage barriers are told to expect an arrival nobody makes and
    the bound is shortened to 2^16 polls; every contraction gives up at its first wait, drains and returns."""
    import numpy as np
    import torch
    from paper_2604_27476_b200 import DecodeContext, EdgefmError, Status, edgefm_debug_set_prefill_wait, edgefm_sync_status
    cfg = CONFIGS["tiny"]
    pair = Pair(cfg, cache_len=4, max_context=64)
    try:
        stream = torch.cuda.current_stream().cuda_stream
        toks = np.random.default_rng(3).integers(0, cfg.vocab, 40).tolist()
        for i, t in enumerate(toks):
            ref, _ = pair.oracle.step(t, 4 + i)
        with pytest.raises(EdgefmError):                           # limits are validated
            edgefm_debug_set_prefill_wait(pair.ctx.handle, 10, 0)
        edgefm_debug_set_prefill_wait(pair.ctx.handle, 1 << 16, 1)
        t0 = time.perf_counter()
        pair.ctx.prefill(toks, 4)
        with pytest.raises(EdgefmError) as ei:
            edgefm_sync_status(pair.ctx.handle, stream)
        dt = time.perf_counter() - t0
        assert ei.value.status == Status.ERR_TIMEOUT
        assert dt < 5.0                                            # five contractions, each gave up within milliseconds
        # the CUDA context is intact: a fresh edgefm context on the same weights prefills the same prompt correctly
        other = DecodeContext(cfg, pair.ptrs, 64)
        other.prefill_kv(pair.kd, pair.vd)
        other.prefill(toks, 4)
        torch.cuda.synchronize()
        other.sync_status()
        assert_logits_close(other.logits.cpu().numpy(), ref, "fresh context after the expired waits")
        other.close()
    finally:
        pair.close()


#: what gives up: (changes to the tiny shape, prompt, cache format)
GIVE_UP = {
    "tiles": (dict(), 40, None),
    "tiles_int8": (dict(), 40, "int8"),
    "persistent": (dict(ffn=9480, n_layers=1, vocab=500), 300, None),
    "pairs": (dict(hidden=3072, n_q_heads=1, n_kv_heads=1, ffn=1872, n_layers=1, vocab=500), 858, None),     # seven row tiles: the last pair has one
    "pairs_few_k_blocks": (dict(hidden=64, ffn=2560, n_layers=1, vocab=500), 421, None),                     # all of K in the ring at once
}


def gives_up_as(cfg, n):
    """The (cluster, pairs) of the shape's contractions with n tokens."""
    from paper_2604_27476_b200 import edgefm_debug_prefill_launch
    from test_prefill_plan import shapes
    return {edgefm_debug_prefill_launch(epi, n, N, K)[2:4] for epi, N, K in shapes(cfg).values()}


@pytest.mark.parametrize("polls", [1024, 1 << 16])
@pytest.mark.parametrize("name", list(GIVE_UP))
def test_a_prompt_cta_that_gives_up_waits_for_its_copies(name, polls):
    """Contractions and attention whose first wait runs out, the producing thread long done with its part (few k-blocks) or stopped by its
    ring: the copies under way must land before the CTA's shared memory is someone else's.  Other contexts, whose kernels follow at once
    on the same stream, compute what they always do, to the bit."""
    import numpy as np
    import torch
    from edgefm_synth import make_weights
    from paper_2604_27476_b200 import DecodeContext, EdgefmError, Status, edgefm_debug_set_prefill_wait, upload_weights
    more, n, kv_format = GIVE_UP[name]
    cfg = CONFIGS["tiny"].with_(qkv_bias=True, **more)
    plans = gives_up_as(cfg, n)
    assert any(c > 0 for c, _ in plans) if name.startswith("tiles") else (0, int(name.startswith("pairs"))) in plans
    ptrs, keep = upload_weights(make_weights(cfg))
    toks = np.random.default_rng(5).integers(0, cfg.vocab, n).tolist()
    ctx, *others = [DecodeContext(cfg, ptrs, n, kv_format=kv_format) for _ in range(4)]
    try:
        others[0].prefill(toks, 0)
        torch.cuda.synchronize()
        others[0].sync_status()
        want = others[0].logits.cpu()
        others[0].append_kv(0)
        edgefm_debug_set_prefill_wait(ctx.handle, polls, 1)
        t0 = time.perf_counter()
        ctx.prefill(toks, 0)
        for o in others:
            o.prefill(toks, 0)
        torch.cuda.synchronize()
        assert time.perf_counter() - t0 < 5.0
        with pytest.raises(EdgefmError) as ei:
            ctx.sync_status()
        assert ei.value.status == Status.ERR_TIMEOUT
        for o in others:
            o.sync_status()
            assert torch.equal(o.logits.cpu(), want)
    finally:
        for c in (ctx, *others):
            c.close()
