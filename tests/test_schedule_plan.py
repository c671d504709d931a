"""The step kernel's plan (no GPU needed): how rows, columns and cached positions are cut, with the arithmetic the kernel itself uses.  Every CTA's
chunks must cover its part of every weight matrix exactly once, stay inside a head, fit the ring and the list, and ask for no box the
tensor maps cannot describe."""
import numpy as np
import pytest

from edgefm_synth import CONFIGS
from paper_2604_27476_b200 import edgefm_debug_step_plan

QKV, O, GU, DN, LM = range(5)
BOX = 255


def shape_of(L=1, H=64, nq=2, nkv=1, d=64, F=64, V=64):
    return dict(n_layers=L, hidden=H, n_q_heads=nq, n_kv_heads=nkv, head_dim=d, ffn=F, vocab=V, rms_eps=1e-6, rope_theta=1e6, qkv_bias=0)


def config_shape(cfg):
    return shape_of(cfg.n_layers, cfg.hidden, cfg.n_q_heads, cfg.n_kv_heads, cfg.head_dim, cfg.ffn, cfg.vocab)


def check_plan(sh, max_context=4096, kv_format="bf16", tokens=1, n_sms=148, ctas=None):
    plan = edgefm_debug_step_plan(sh, max_context, kv_format, tokens, n_sms)
    H, F, V, d, nq, nkv = sh["hidden"], sh["ffn"], sh["vocab"], sh["head_dim"], sh["n_q_heads"], sh["n_kv_heads"]
    units = [(nq + 2 * nkv) * d // 2, H, F, H, V]
    G = plan["ctas"]
    assert G == min(n_sms, H)
    assert plan["dynamic_smem_bytes"] <= 232448 and plan["ring_bytes"] >= plan["max_chunk_bytes"]
    assert plan["max_chunk_bytes"] >= plan["kv_block"] * d * (4 if kv_format == "bf16" else 2)
    assert plan["merged_len"] * G >= nq * d and (plan["tight"] or plan["merged_len"] <= 128)
    listed = np.zeros(G, np.int64)
    for op in range(5):
        cols, K = plan["cols"][op], plan["cols"][op]["K"]
        assert K == (nq * d if op == O else F if op == DN else H)
        assert (cols["segs"] - 1) * cols["seg"] < K <= cols["segs"] * cols["seg"]
        if cols["box_rows"]:
            assert K % 64 == 0 and cols["seg"] % 64 == 0 and cols["box_rows"] <= 256 and cols["seg"] // 64 <= 256
        covered = np.zeros(units[op], np.int64)
        for c in range(G) if ctas is None else sorted({c for c in ctas if c < G} | {G - 1}):
            _, chunks = edgefm_debug_step_plan(sh, max_context, kv_format, tokens, n_sms, op=op, cta=c)
            listed[c] += len(chunks)
            at, u1 = units[op] * c // G, units[op] * (c + 1) // G
            for i, (x, y, z, w, u, n) in enumerate(chunks.astype(np.int64)):
                seg = i % cols["segs"]
                assert u == at and n >= 1 and u + n <= u1 and n <= cols["tile"]
                paired = op in (QKV, GU)
                assert (y == 0xffffffff) == (not paired)
                if op == QKV:
                    assert u // (d // 2) == (u + n - 1) // (d // 2)
                row = u // (d // 2) * d + u % (d // 2) if op == QKV else u
                partner = row + (d // 2 if op == QKV else F)
                how = w >> 16
                if how == BOX:
                    assert x == row and (not paired or y == partner) and (w & 0xffff) * 64 == seg * cols["seg"] and n <= cols["box_rows"]
                    part = z
                    assert part == cols["box_rows"] * cols["seg"] * 2
                else:
                    assert x * 8 == row * K + seg * cols["seg"] and (not paired or y * 8 == partner * K + seg * cols["seg"])
                    assert how == (n if cols["segs"] > 1 else 0)
                    part = z * max(how, 1)
                    assert part == n * min(cols["seg"], K - seg * cols["seg"]) * 2
                assert part * (2 if paired else 1) <= plan["max_chunk_bytes"]
                if seg == cols["segs"] - 1:
                    covered[u:u + n] += 1
                    at = u + n
            assert at == u1
        if ctas is None:
            assert (covered == 1).all()
    assert plan["tight"] or listed.max() <= plan["list_len"]
    return plan


@pytest.mark.parametrize("name", sorted(CONFIGS))
@pytest.mark.parametrize("tokens", [1, 2, 4, 8])
def test_schedule_covers_every_weight_exactly_once(name, tokens):
    for n_sms in (148, 132, 16):
        if tokens == 8 and n_sms < 148:        # (a shape that does not fit the eight-token build is verified by the prompt kernels)
            continue
        plan = check_plan(config_shape(CONFIGS[name]), tokens=tokens, n_sms=n_sms, ctas=None if n_sms == 16 else range(0, 148, 7))
        if n_sms == 148:
            assert not plan["tight"] and plan["kv_block"] == 128 // (CONFIGS[name].head_dim // 64)


def test_schedule_odd_shapes_and_small_grids():
    for sh in (shape_of(H=72, F=40, V=1), shape_of(H=2200, F=1400, V=301), shape_of(H=4168, nq=7, F=72), shape_of(H=888, F=6104, V=152064),
               shape_of(H=136, nq=40, nkv=8, d=128, V=103000)):
        for tokens in (1, 2, 4):
            for n_sms in (5, 148):
                check_plan(sh, tokens=tokens, n_sms=n_sms)


# Many heads on few rows; vectors of 16 - 31 thousand values; long vocabularies on short rows: shapes the usual layout has no room for must be laid out
# in a tight build, not refused.
TIGHT = {
    "few_rows_many_heads": (shape_of(80, 8, 44, 22, 128, 40, 101), 64, "int8", 1),
    "few_rows_many_heads_4": (shape_of(24, 8, 12, 3, 128, 256, 438), 4096, "bf16", 4),
    "few_rows_long_vocabulary": (shape_of(1, 8, 32, 4, 128, 15624, 699941), 4096, "int8", 1),
    "outputs_24576": (shape_of(1, 152, 192, 24, 128, 1536, 113), 64, "bf16", 1),
    "hidden_13800": (shape_of(80, 13800, 135, 27, 128, 808, 7), 4096, "bf16", 1),
    "hidden_23960": (shape_of(80, 23960, 18, 6, 64, 1448, 59), 20000, "bf16", 1),
    "hidden_24056": (shape_of(24, 24056, 8, 4, 64, 160, 34), 4096, "int8", 1),
    "hidden_26280": (shape_of(1, 26280, 12, 2, 64, 3960, 7), 64, "int8", 1),
    "hidden_30640": (shape_of(1, 30640, 4, 2, 64, 64, 32), 64, "int8", 1),
}


@pytest.mark.parametrize("name", sorted(TIGHT))
def test_shapes_that_leave_little_room(name):
    sh, max_context, kv_format, tokens = TIGHT[name]
    assert check_plan(sh, max_context, kv_format, tokens, ctas=(0, 1, 63))["tight"]


def test_matrices_past_the_offsets_of_a_chunk_are_refused():
    """Offsets are 32 bits of 16-byte units: the last row of a 64 GiB matrix is in reach, one of a larger matrix would be taken from its start."""
    from paper_2604_27476_b200 import EdgefmError, Status
    last = 2 ** 32 // 300                                         # rows of 2400 columns
    _, chunks = edgefm_debug_step_plan(shape_of(H=2400, V=last), 64, op=LM, cta=147)
    x, _, z, _, u, n = chunks[-1].astype(np.int64)
    assert u + n == last and x == u * 300 and z == n * 4800
    with pytest.raises(EdgefmError) as ei:
        edgefm_debug_step_plan(shape_of(H=2400, V=last + 1), 64)
    assert ei.value.status == Status.ERR_BAD_SHAPE and "64 GiB" in str(ei.value)
    with pytest.raises(EdgefmError):
        edgefm_debug_step_plan(shape_of(H=2400, F=last // 2 // 8 * 8 + 8), 64)      # gate and up rows are one matrix


def test_what_gives_way():
    """In order: tables and lists, chunk sizes, the cached positions of a chunk."""
    far = edgefm_debug_step_plan(shape_of(H=24056, nq=4, nkv=4, F=160, V=300), 4096)
    assert far["tight"] and far["unit_table_bytes"] > 0 and far["max_chunk_bytes"] > 33 * 1024 and far["kv_block"] == 128
    small = edgefm_debug_step_plan(shape_of(H=28800, nq=4, nkv=4, F=64, V=300), 4096)
    assert small["tight"] and small["max_chunk_bytes"] <= 32 * 1024 + 128 and small["kv_block"] == 128
    half = edgefm_debug_step_plan(shape_of(H=15616, nq=8, nkv=4, d=128, F=64, V=300), 4096, tokens=2)
    assert half["tight"] and half["max_chunk_bytes"] <= 16 * 1024 + 128 and half["kv_block"] == 32
