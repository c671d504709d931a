"""The work a user of this library has it do, as measurable cases: greedy decoding, verification of proposed blocks and prompt
processing, each through the public binding (`DecodeContext`), for the Qwen2.5-style shapes this repository is built for.

A case is a dict of plain values; `listed()` gives the standing ones, `draw()` more of the same ranges.  Common fields:

  path     "decode"  : `steps` chained greedy steps behind a cache of `context` positions
           "verify"  : `rounds` proposed blocks of `block` tokens, each followed by the read-back of the cache length
           "prefill" : a prompt of `prompt` tokens behind a kept prefix of `context` positions
  model    one of MODELS
  kv       cache format, "bf16" or "int8"
  subset   decode only: output layer pruned to that many token ids (0 = the whole vocabulary)
  build    verify only: block_tokens of the context (4: the step kernel carries the block; 0: a plain context)

A pass first drops what the previous pass left behind the kept prefix (`append_kv(context)`), which is how a request slot with a
fixed prefix is reused.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import torch

from paper_2604_27476_b200.binding import DecodeContext


def _model(n_layers, hidden, n_q_heads, n_kv_heads, head_dim, ffn, vocab, qkv_bias=True, tied=False):
    return SimpleNamespace(n_layers=n_layers, hidden=hidden, n_q_heads=n_q_heads, n_kv_heads=n_kv_heads, head_dim=head_dim, ffn=ffn,
                           vocab=vocab, qkv_bias=qkv_bias, tied=tied, rms_eps=1e-6, rope_theta=1e6)


#: The shapes of this repository's configurations.
MODELS = {
    "tiny": _model(2, 256, 4, 2, 64, 688, 4096, qkv_bias=False),
    "qwen2.5-0.5b": _model(24, 896, 14, 2, 64, 4864, 151936, tied=True),
    "qwen2.5-1.5b": _model(28, 1536, 12, 2, 128, 8960, 151936),
    "qwen2.5-3b": _model(36, 2048, 16, 2, 128, 11008, 151936),
    "qwen2.5-7b": _model(28, 3584, 28, 4, 128, 18944, 152064),
}

#: Rows of the output matrix that stand for frequent tokens.  A trained model's next-token distribution is peaked: its two largest
#: logits are about one apart.  Independent rows of one size would leave them 0.1 apart, closer than any two models' would be.
FREQUENT = 64


def listed():
    return [
        # The smallest call there is: two small layers, all of it in L2; latency, launches and synchronisation only.
        dict(name="decode-tiny", path="decode", model="tiny", context=128, steps=8, kv="bf16", subset=0),
        # A small vision-language assistant: 256 of the cached positions are image tokens.
        dict(name="decode-0.5b", path="decode", model="qwen2.5-0.5b", context=1024, steps=8, kv="bf16", subset=0),
        # The ordinary decode loop at the headline shape and context.
        dict(name="decode-1.5b", path="decode", model="qwen2.5-1.5b", context=2048, steps=8, kv="bf16", subset=0),
        # A short dialogue turn on a task-specific build whose vocabulary is pruned.
        dict(name="decode-1.5b-subset", path="decode", model="qwen2.5-1.5b", context=337, steps=8, kv="bf16", subset=32768),
        # Long documents: a 32k cache at the largest shape.
        dict(name="decode-7b-32k", path="decode", model="qwen2.5-7b", context=32768, steps=4, kv="bf16", subset=0),
        # A long session whose cache is kept compressed to save memory.
        dict(name="decode-3b-int8", path="decode", model="qwen2.5-3b", context=9001, steps=4, kv="int8", subset=0),
        # Speculative decoding, the base model's side: blocks of four on a context built for them.
        dict(name="verify-4", path="verify", model="qwen2.5-1.5b", context=2048, block=4, build=4, rounds=4, kv="bf16"),
        # The same with blocks of eight on a plain context.
        dict(name="verify-8", path="verify", model="qwen2.5-1.5b", context=2048, block=8, build=0, rounds=4, kv="bf16"),
        # A user's short question behind a system prompt and image whose cache rows are kept.
        dict(name="prefill-0.5b-suffix", path="prefill", model="qwen2.5-0.5b", context=1024, prompt=77, kv="bf16"),
        # The prompt of the headline shape.
        dict(name="prefill-1.5b", path="prefill", model="qwen2.5-1.5b", context=0, prompt=2048, kv="bf16"),
        # A page of text into a compressed cache.
        dict(name="prefill-3b-int8", path="prefill", model="qwen2.5-3b", context=0, prompt=1000, kv="int8"),
        # A document at the largest shape, longer than one pass of the dense path.
        dict(name="prefill-7b", path="prefill", model="qwen2.5-7b", context=0, prompt=4200, kv="bf16"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: model, option and sizes over the ranges of the listed ones (sizes spread over their logarithm)."""
    path = rng.choice(["decode", "decode", "verify", "prefill", "prefill"])
    model = rng.choice([m for m in MODELS if m != "tiny"])
    if path == "decode":
        if rng.random() < 0.15:
            model = "tiny"
        kv = "int8" if rng.random() < 0.25 else "bf16"
        subset = _log_int(rng, 500, min(65536, MODELS[model].vocab // 2)) if rng.random() < 0.25 else 0
        return dict(path=path, model=model, context=_log_int(rng, 100, 32768), steps=rng.randint(2, 8 if model != "qwen2.5-7b" else 4), kv=kv,
                    subset=subset)
    if path == "verify":
        block = rng.randint(2, 8)
        return dict(path=path, model=model, context=_log_int(rng, 100, 8000), block=block, build=4 if block <= 4 else 0, rounds=rng.randint(1, 4),
                    kv="bf16")
    most = work(listed()[-1])["flops"]
    while True:
        case = dict(path=path, model=model, context=rng.choice([0, _log_int(rng, 32, 4096)]), prompt=_log_int(rng, 9, 8192),
                    kv="int8" if rng.random() < 0.25 else "bf16")
        if work(case)["flops"] <= most:
            return case


def _weights(m, gen, dev):
    """bf16 weights on the device: matrices and biases N(0, 0.02), norm weights around one."""
    keep = []

    def normal(*shape, std=0.02, mean=0.0):
        t = torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(mean, std, generator=gen)
        keep.append(t)
        return t

    r, qd = (m.n_q_heads + 2 * m.n_kv_heads) * m.head_dim, m.n_q_heads * m.head_dim
    layers = []
    for _ in range(m.n_layers):
        layers.append({
            "input_norm": normal(m.hidden, std=0.1, mean=1.0).data_ptr(),
            "wqkv": normal(r, m.hidden).data_ptr(),
            "bqkv": normal(r).data_ptr() if m.qkv_bias else None,
            "wo": normal(m.hidden, qd).data_ptr(),
            "post_norm": normal(m.hidden, std=0.1, mean=1.0).data_ptr(),
            "w_gate_up": normal(2 * m.ffn, m.hidden).data_ptr(),
            "w_down": normal(m.hidden, m.ffn).data_ptr(),
        })
    ranked = torch.randperm(m.vocab, generator=gen, device=dev)      # token ids, the frequent ones first
    embed = normal(m.vocab, m.hidden)
    lm_head = embed if m.tied else normal(m.vocab, m.hidden)
    lm_head[ranked[:FREQUENT]] *= 4
    pointers = {"embed": embed.data_ptr(), "final_norm": normal(m.hidden, std=0.1, mean=1.0).data_ptr(), "lm_head": lm_head.data_ptr(),
                "layers": layers}
    return pointers, keep, ranked


def prepare(case, seed):
    m = MODELS[case["model"]]
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    pointers, keep, ranked = _weights(m, gen, dev)
    path, context, rounds = case["path"], case["context"], case.get("rounds", 0)
    # the rows a pass adds; a prompt fills its cache exactly, so that the whole cache is the result
    added = case["steps"] if path == "decode" else rounds * case["block"] if path == "verify" else case["prompt"]
    ctx = DecodeContext(m, pointers, context + added, kv_format=case["kv"], block_tokens=case.get("build", 0))
    if context:
        # the kept prefix, as an earlier request left it
        shape = (m.n_layers, m.n_kv_heads, context, m.head_dim)
        k = torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(generator=gen)
        v = torch.empty(shape, dtype=torch.bfloat16, device=dev).normal_(generator=gen)
        ctx.prefill_kv(k, v)
        torch.cuda.current_stream().synchronize()
    state = SimpleNamespace(case=case, ctx=ctx, keep=keep, logits=ctx.logits, out=None)
    if case.get("subset"):
        ctx.set_vocab_subset(ranked[: case["subset"]].sort().values.cpu().numpy())
        state.logits = ctx.logits[: case["subset"]]
    n_tokens = {"decode": 1, "verify": rounds * case.get("block", 0), "prefill": case.get("prompt", 0)}[path]
    tokens = torch.randint(m.vocab, (n_tokens,), generator=gen, device=dev).tolist()
    if path == "verify":
        # (a step costs the same whether its proposals are accepted or not)
        state.blocks = [tokens[i * case["block"]: (i + 1) * case["block"]] for i in range(rounds)]
        state.logits = ctx.block_logits[: case["block"]]
    elif path == "decode":
        state.token = tokens[0]
        # an image of 16 x 16 tokens advances the rotary position by 16 instead of 256
        state.position = context - 240 if case["model"] == "qwen2.5-0.5b" and context >= 256 else context
    else:
        state.tokens = tokens
    return state


def run(state):
    case, ctx = state.case, state.ctx
    ctx.append_kv(case["context"])          # back to the kept prefix
    if case["path"] == "decode":
        ctx.step(state.token, state.position)
        for _ in range(case["steps"] - 1):
            ctx.step()                      # chained on the device
        return {"logits": state.logits, "next_token": ctx.next_token}
    if case["path"] == "verify":
        lengths = [case["context"]]
        for block in state.blocks:
            ctx.verify_block(block, lengths[-1])
            lengths.append(ctx.sync_length())   # what the next proposal starts from
        return {"logits": state.logits, "n_accepted": ctx.n_accepted, "next_token": ctx.next_token, "lengths": lengths}
    ctx.prefill(state.tokens, case["context"])
    out = {"logits": state.logits, "next_token": ctx.next_token}
    if case["kv"] == "bf16":
        # the rows the prompt is processed for, as another slot takes them over
        k, v = ctx.export_kv()
        out["k"], out["v"] = k.view(torch.bfloat16), v.view(torch.bfloat16)
    return out


def work(case):
    """Weights once per step, block or prompt; cached rows read once, new rows written once; the logits."""
    m = MODELS[case["model"]]
    r, qd = (m.n_q_heads + 2 * m.n_kv_heads) * m.head_dim, m.n_q_heads * m.head_dim
    per_layer = r * m.hidden + m.hidden * qd + 3 * m.ffn * m.hidden
    vectors = m.n_layers * (2 * m.hidden + (r if m.qkv_bias else 0)) + m.hidden
    out_rows = case.get("subset") or m.vocab
    head = m.head_dim * 2 if case["kv"] == "bf16" else m.head_dim + 4
    row = 2 * m.n_layers * m.n_kv_heads * head                       # K and V of one position, all layers
    context = case["context"]

    def one(n, start, logit_rows):
        """n tokens together behind `start` cached positions."""
        weights = 2 * (m.n_layers * per_layer + vectors + out_rows * m.hidden + n * m.hidden)
        nbytes = weights + row * (start + n) + 4 * out_rows * logit_rows
        pairs = n * start + n * (n + 1) // 2
        flops = 2 * n * m.n_layers * per_layer + 4 * pairs * qd * m.n_layers + 2 * out_rows * m.hidden * logit_rows
        return nbytes, flops

    if case["path"] == "decode":
        parts = [one(1, context + i, 1) for i in range(case["steps"])]
    elif case["path"] == "verify":
        parts = [one(case["block"], context, case["block"]) for _ in range(case["rounds"])]
    else:
        parts = [one(case["prompt"], context, 1)]
        if case["kv"] == "bf16":
            parts.append((2 * row * (context + case["prompt"]), 0))   # the exported copy: read and written
    return {"bytes": sum(p[0] for p in parts), "flops": sum(p[1] for p in parts)}


def tolerance(case):
    """Decode: fp32 sums of 24-bit activations, but a new cache row is rounded to bf16 (or 8-bit codes), and a value that straddles a
    rounding boundary moves what follows.  Blocks of more than two tokens and prompts multiply 16-bit activations, and a prompt's
    rows come back as bf16."""
    if case["path"] == "prefill":
        return {"rel": 5e-3, "max": 5e-2}
    if case["path"] == "verify":
        return {"rel": 2e-3, "max": 2e-2}
    return {"rel": 1e-3, "max": 1e-2} if case["kv"] == "int8" else {"rel": 2e-4, "max": 2e-3}
