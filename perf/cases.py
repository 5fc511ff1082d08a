"""The work that a user of the library has it do, as cases that can be timed.

Two kinds of pass.  A *step* is one denoising step of a model's attention path through the public entry points, in the
order in which a generation loop calls them: for every layer `ec_attend` (fresh K/V rows into the cache, then the active
rows attend over it), one gate call over the step's logits, one selection of the next step's rows.  `rows = "skip"` is
the partial step (the block's mask tokens and the k most recently decoded ones are the queries), `rows = "full"` the
recomputation, in which every position is.  A *gate* pass is the gate alone, as a program calls it that keeps its own
attention.  Every buffer, row list, workspace and descriptor that such a loop keeps from step to step is made by
`prepare`.
"""
import math

import numpy as np
import torch

import paper_2603_18489_b200 as ec

TAU = 1.5              # nats
CONF_THRESHOLD = 0.9   # confidence above which a masked row is decoded

LLADA = dict(dtype="bf16", q_heads=32, kv_heads=32, head_dim=128, vocab=126464)
DREAM = dict(dtype="bf16", q_heads=28, kv_heads=4, head_dim=128, vocab=152064)


def _step(name, rows, model, *, batch=1, ctx, block=32, k, layers, loop="block", refresh="fused", score_std=1.0):
    """`loop`: block-wise decoding with the decoded flags given, or a sliding window with the decoding inside the gate.
    `refresh`: the cache update inside ec_attend, or as a call of its own in front of it.  `score_std`: standard
    deviation of the attention scores (1: flat softmax rows; 4: rows ruled by a few keys)."""
    return dict(model, name=name, kind="step", rows=rows, batch=batch, ctx=ctx, block=block, k=k, layers=layers,
                loop=loop, refresh=refresh, score_std=float(score_std))


def _gate(name, entry, dtype, *, batch, block, vocab, pad=0):
    """`pad`: columns behind the vocabulary in every row of the logits."""
    return dict(name=name, kind="gate", entry=entry, dtype=dtype, batch=batch, block=block, vocab=vocab, pad=pad)


def listed():
    return [
        # the repository's first configuration: one fp32 layer, four heads of 64; every launch is a handful of blocks
        _step("tiny_f32_skip", "skip", dict(dtype="f32", q_heads=4, kv_heads=4, head_dim=64, vocab=1024),
              ctx=256, k=2, layers=1),
        # the usual partial step at a short context, whole model, both model geometries and both ways of decoding
        _step("llada_768_skip", "skip", LLADA, ctx=768, k=2, layers=32),
        _step("dream_768_skip", "skip", DREAM, ctx=768, k=8, layers=28, loop="sliding"),
        # a long prompt at the paper's default budget of recent tokens; a length that no tile divides, peaky attention
        _step("llada_1983_skip_k64", "skip", LLADA, ctx=1983, k=64, layers=32, loop="sliding", score_std=4.0),
        # the benchmark's headline step
        _step("llada_4096_skip", "skip", LLADA, ctx=4096, k=2, layers=32),
        # eight sequences served together; a slice of the layers, as all of them only repeat it
        _step("llada_4096_b8_skip", "skip", LLADA, batch=8, ctx=4096, k=2, layers=4),
        # heads of 64 in bf16, grouped queries, four sequences, the cache update called by itself
        _step("d64_1000_b4_skip", "skip", dict(dtype="bf16", q_heads=12, kv_heads=4, head_dim=64, vocab=32000),
              batch=4, ctx=1000, k=16, layers=12, refresh="separate"),
        # recomputation: the short context, two ragged sequences with grouped queries, and the largest one
        _step("llada_768_full", "full", LLADA, ctx=768, k=2, layers=32),
        _step("dream_1531_b2_full", "full", DREAM, batch=2, ctx=1531, k=8, layers=14, loop="sliding", score_std=4.0),
        _step("llada_4096_b8_full", "full", LLADA, batch=8, ctx=4096, k=2, layers=2),
        # the gate alone: eight sequences of bf16 logits, and fp32 logits of an odd vocabulary in padded rows
        _gate("gate_bf16_b8", "decode", "bf16", batch=8, block=32, vocab=126464),
        _gate("gate_f32_odd", "metrics", "f32", batch=1, block=32, vocab=32001, pad=7),
    ]


# ------------------------------------------------------------------------------------------------------- drawn cases
MOST_FLOPS = 4 * 2 * 8 * 32 * 4096 ** 2 * 128   # of llada_4096_b8_full
MOST_BYTES = 3e9                                # of caches, activations and logits in one state


def _log_int(rng, lo, hi):
    return min(hi, int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1)))))


def draw(rng):
    kind = rng.choice(["skip", "skip", "skip", "full", "full", "gate"])
    if kind == "gate":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        vocab = rng.choice([126464, 152064, _log_int(rng, 1024, 160000)])
        pad = -vocab % 8 + 8 * rng.randint(0, 2)
        return _unnamed(_gate("", rng.choice(["flags", "decode", "metrics"]), dtype, batch=_log_int(rng, 1, 8),
                              block=rng.choice([8, 16, 32, 32, 64]), vocab=vocab, pad=pad))
    full = kind == "full"
    size = rng.random()
    if size < 0.8:
        model, depth = (LLADA, 32) if size < 0.4 else (DREAM, 28)
        batch = rng.choice([1, 1, 1, _log_int(rng, 2, 8)])
        ctx = _log_int(rng, 256, 4096)
        refresh = "fused"
    else:
        groups = rng.choice([1, 1, 2, 3])
        kv = rng.choice([2, 4, 8])
        model = dict(dtype=rng.choice(["bf16", "bf16", "f32"]), q_heads=kv * groups, kv_heads=kv,
                     head_dim=64, vocab=_log_int(rng, 1024, 40000) // 8 * 8)
        depth = 12
        batch = _log_int(rng, 1, 4)
        ctx = _log_int(rng, 192, 512 if full and model["dtype"] == "f32" else 1024)
        refresh = rng.choice(["fused", "separate"])
    case = _step("", kind, model, batch=batch, ctx=ctx, k=rng.choice([0] + 4 * [_log_int(rng, 1, 64)]),
                 layers=1, loop=rng.choice(["block", "sliding"]), refresh=refresh, score_std=rng.choice([1.0, 1.0, 4.0]))
    one = work(case)
    w = dict(case, layers=2)
    most = min(depth, int((MOST_BYTES - one["bytes"]) / (work(w)["bytes"] - one["bytes"])),
               int(MOST_FLOPS / max(1, work(w)["flops"] - one["flops"])))
    case["layers"] = max(1, min(most, _log_int(rng, 2, depth)))
    return _unnamed(case)


def _unnamed(case):
    return {key: value for key, value in case.items() if key != "name"}


# ------------------------------------------------------------------------------------------------------------ inputs
def _rows(case):
    return case["ctx"] if case["rows"] == "full" else case["block"] + case["k"]


def _logits(g, rows, vocab, pad, dtype):
    """Rows from flat to peaked, as the model's certainty about a position goes; nothing may read the padding."""
    sigma = torch.rand(rows, 1, generator=g, device="cuda") * 7.5 + 0.5
    x = torch.randn(rows, vocab + pad, generator=g, device="cuda") * sigma
    x[:, vocab:] = 1e4
    return x.to(dtype)


def _flags(rng, batch, block):
    """Half of each block's rows newly decoded."""
    f = np.zeros((batch, block), np.uint8)
    for b in range(batch):
        f[b, rng.choice(block, size=block // 2, replace=False)] = 1
    return f.reshape(-1)


def _gate_buffers(state, batch, block, vocab):
    n = batch * block
    i32 = dict(dtype=torch.int32, device="cuda")
    f32 = dict(dtype=torch.float32, device="cuda")
    state.update(gate_ws=ec.new_workspace(ec.ec_entropy_gate_workspace_bytes(n, vocab)),
                 gate_out=dict(argmax_out=torch.zeros(n, **i32), conf_out=torch.zeros(n, **f32),
                               entropy_out=torch.zeros(n, **f32), max_entropy_out=torch.zeros(batch, **f32),
                               decision_out=torch.zeros(batch, **i32)),
                 decoded=torch.zeros(n, dtype=torch.uint8, device="cuda"),
                 row_mask=torch.ones(n, dtype=torch.uint8, device="cuda"), tokens=torch.full((n,), -1, **i32))


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    rng = np.random.default_rng(int(seed))
    dtype = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    batch, block, vocab = case["batch"], case["block"], case["vocab"]
    state = dict(case=case, logits=_logits(g, batch * block, vocab, case.get("pad", 0), dtype),
                 flags=torch.from_numpy(_flags(rng, batch, block)).cuda())
    _gate_buffers(state, batch, block, vocab)
    if case["kind"] == "gate":
        return state

    ctx, k, layers = case["ctx"], case["k"], case["layers"]
    hq, hkv, d, n = case["q_heads"], case["kv_heads"], case["head_dim"], _rows(case)

    def normal(std, *shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=dtype).mul_(std)

    std = math.sqrt(case["score_std"])
    q, k_new, v_new = normal(std, layers, batch, n, hq, d), normal(std, layers, batch, n, hkv, d), normal(1.0, layers, batch, n, hkv, d)
    k_cache, v_cache = normal(std, layers, batch, hkv, ctx, d), normal(1.0, layers, batch, hkv, ctx, d)
    out = torch.zeros_like(q)
    # with several layers the call before an ec_attend works on another layer's caches
    desc = ec.make_desc(batch, ctx, hq, hkv, d, dtype, flags=ec.EC_ATTN_CACHE_SETTLED if layers > 1 else 0)

    # The loop in the middle of the generation: half the context is prompt, half of the rest is decoded, the window
    # follows.  Decoded positions carry the step that decoded them, a few of them each step.
    start = max(k, min(ctx - block, ctx // 2 + (ctx - ctx // 2) // 2))
    prompt = min(ctx // 2, start - k)
    steps = max(1, (start - prompt) // 3)
    history = np.full((batch, ctx), ec.EC_H_NEVER, np.int32)
    rows = np.empty((batch, block + k), np.int32)
    for b in range(batch):
        history[b, prompt:start] = 1 + np.minimum(np.arange(start - prompt) // 3, steps - 1)
        recent = rng.choice(np.arange(max(prompt, start - 4 * k - 8), start), size=k, replace=False)
        rows[b] = np.concatenate([np.arange(start, start + block), np.sort(recent)])
    next_rows = np.full((batch, block + k + 8), -1, np.int32)
    next_rows[:, :block] = np.arange(start, start + block)
    masked = np.zeros((batch, ctx), np.uint8)
    masked[:, start:] = 1
    loop = ec.new_step_state(batch, steps + 1)
    loop[:, 1:3] = torch.tensor([4, 1], dtype=torch.int32, device="cuda")
    state.update(desc=desc, q=q, out=out, k_cache=k_cache, v_cache=v_cache,
                 layer=[tuple(t[i] for t in (q, k_new, v_new, k_cache, v_cache, out)) for i in range(layers)],
                 rows=None if case["rows"] == "full" else torch.from_numpy(rows).cuda(),
                 attend_ws=ec.new_workspace(ec.ec_attend_workspace_bytes(desc, n)),
                 history=torch.from_numpy(history).cuda(), loop=loop, masked=torch.from_numpy(masked).cuda(),
                 window_start=torch.full((batch,), start, dtype=torch.int32, device="cuda"),
                 next_rows=torch.from_numpy(next_rows).cuda())
    return state


# -------------------------------------------------------------------------------------------------------------- pass
def _run_gate(s):
    case = s["case"]
    entry, vocab, block = case["entry"], case["vocab"], case["block"]
    if entry == "metrics":
        return ec.ec_entropy_gate_metrics(s["logits"], vocab, block, s["flags"], TAU, workspace=s["gate_ws"])
    if entry == "flags":
        return ec.ec_entropy_gate(s["logits"], vocab, block, s["flags"], TAU, workspace=s["gate_ws"], **s["gate_out"])
    s["row_mask"].fill_(1)      # every row of a window is a mask token, each step anew
    got = ec.ec_entropy_gate_decode(s["logits"], vocab, block, s["row_mask"], CONF_THRESHOLD, TAU, s["tokens"],
                                    decoded_out=s["decoded"], workspace=s["gate_ws"], **s["gate_out"])
    return dict(got, masked=s["row_mask"], tokens=s["tokens"])


def run(state):
    s = state
    case = s["case"]
    if case["kind"] == "gate":
        return _run_gate(s)
    desc, rows, ws = s["desc"], s["rows"], s["attend_ws"]
    if case["refresh"] == "separate":
        for q, k_new, v_new, k_cache, v_cache, out in s["layer"]:
            ec.ec_kv_refresh(desc, k_cache, v_cache, k_new, v_new, rows)
            ec.ec_attend(desc, q, None, None, k_cache, v_cache, rows, out=out, workspace=ws)
    else:
        for q, k_new, v_new, k_cache, v_cache, out in s["layer"]:
            ec.ec_attend(desc, q, k_new, v_new, k_cache, v_cache, rows, out=out, workspace=ws)
    vocab, block, k = case["vocab"], case["block"], case["k"]
    if case["loop"] == "block":
        gate = ec.ec_entropy_gate(s["logits"], vocab, block, s["flags"], TAU, workspace=s["gate_ws"], **s["gate_out"])
        ec.ec_select_recent(s["history"], s["loop"], s["flags"], s["window_start"], block, gate["decision"], k,
                            s["next_rows"])
    else:
        s["row_mask"].fill_(1)
        gate = ec.ec_entropy_gate_decode(s["logits"], vocab, block, s["row_mask"], CONF_THRESHOLD, TAU, s["tokens"],
                                         decoded_out=s["decoded"], workspace=s["gate_ws"], **s["gate_out"])
        ec.ec_select_recent_sliding(s["history"], s["loop"], s["masked"], gate["decoded"], block, gate["decision"], k,
                                    s["next_rows"])
    return dict(gate=gate, out=s["out"], k_cache=s["k_cache"], v_cache=s["v_cache"], tokens=s["tokens"],
                history=s["history"], loop=s["loop"], masked=s["masked"], next_rows=s["next_rows"])


# ---------------------------------------------------------------------------------------------------------- the floor
def work(case):
    """Logits read once; on a step also, per layer: q read and out written, the fresh rows read and written into the
    cache, the other rows of the cache read; history read and row list written; two products per query, key and head."""
    e = 2 if case["dtype"] == "bf16" else 4
    batch, block, vocab = case["batch"], case["block"], case["vocab"]
    n_bytes = batch * block * (vocab * e + 12)
    if case["kind"] == "gate":
        return {"bytes": n_bytes, "flops": 4 * batch * block * vocab}
    ctx, hq, hkv, d, n = case["ctx"], case["q_heads"], case["kv_heads"], case["head_dim"], _rows(case)
    layer = batch * d * e * (2 * n * hq + 4 * n * hkv + 2 * (ctx - n) * hkv)
    n_bytes += case["layers"] * layer + batch * 4 * (ctx + block + case["k"])
    return {"bytes": n_bytes, "flops": 4 * batch * block * vocab + case["layers"] * 4 * batch * n * ctx * hq * d}


def tolerance(case):
    """Attention in bf16 rounds its probabilities and its results to 8 bits; all else is fp32, whole numbers and bytes."""
    return {"rel": 1e-2 if case["kind"] == "step" and case["dtype"] == "bf16" else 1e-5}
