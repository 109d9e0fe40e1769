"""The work a user of the AG-gated attention layer has it do, as timed cases.

A case is one pass through the public calls of `paper_2410_12876_b200.binding` (and of
`schedule.chained_layer`, for a layer that owns its projections) on buffers that are set up once:

    layer    gate -> compaction -> prefill attention on given Q, K, V, then decode steps
    chain    gate -> Q, K, V projection into the cache -> prefill attention -> output projection with
             the skip connection (the layer of a stack, fed with hidden states only), then decode steps
    attend   compaction -> prefill attention under given flags (a layer that evicts by flags computed
             elsewhere, as under the previous layer's gate)
    decode   decode steps on a cache that is already there, rewound to the end of the prompt first
             (several continuations of one prompt)

Shapes are the repository's own: the Llama-2-7B-shaped layer (hidden 4096, 32 heads x 128, gate
4 x 128), the same with 8 key/value heads, a layer of 64-wide heads, and the float32 correctness layer.
"""
import math

import numpy as np
import torch

from paper_2410_12876_b200 import binding as ag
from paper_2410_12876_b200 import inputs, schedule

# hidden, heads, kv_heads, head_dim, gate_heads, gate_head_dim, dtype
ARCHS = {
    "7b": (4096, 32, 32, 128, 4, 128, "bf16"),
    "gqa": (4096, 32, 8, 128, 4, 128, "bf16"),
    "heads64": (1024, 16, 16, 64, 4, 64, "bf16"),
    "f32": (256, 4, 4, 64, 2, 64, "f32"),
    "f32_wide": (512, 8, 8, 128, 2, 128, "f32"),
}


def _case(name, kind, arch, batch, seq, keep=(0.3, 0.8), gate="global", ragged=False, window=0, steps=0, graph=False,
          empty_heads=0):
    c = {"kind": kind, "arch": arch, "batch": batch, "seq": seq, "keep_lo": keep[0], "keep_hi": keep[1], "gate": gate,
         "ragged": ragged, "window": window, "steps": steps, "graph": graph, "empty_heads": empty_heads}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the float32 correctness layer: every call of the layer at its smallest, prompt and 16 decode steps
        _case("tiny_f32", "layer", "f32", 1, 128, keep=(0.5, 0.5), steps=16),
        # a short prompt of odd length through a whole layer of a stack, then the first tokens of the answer
        _case("short_prompt", "chain", "7b", 1, 333, steps=4),
        # the headline prompt: one 7B-shaped layer, 4096 tokens, keep rates spread over the heads
        _case("prompt_7b", "layer", "7b", 1, 4096),
        # the largest: one layer of the 32-layer stack at batch 8, projections inside the path
        _case("stack_batch8", "chain", "7b", 8, 4096),
        # a deep layer of a long prompt: most tokens evicted, a quarter of the heads keep nothing
        _case("deep_prompt", "attend", "7b", 1, 16384, keep=(0.1, 0.1), empty_heads=8),
        # a batch of documents through the local gate (one linear layer), padded to a common odd length
        _case("local_gate", "layer", "7b", 2, 3001, gate="local", ragged=True),
        # grouped-query layer with a window of recent tokens over a padded batch: prompt and a few steps
        _case("window_gqa", "layer", "gqa", 4, 1999, ragged=True, window=5, steps=4),
        # a batch through a layer of 64-wide heads (head_dim 64 and gate heads of 64)
        _case("heads64", "layer", "heads64", 4, 1500, steps=2),
        # one user's answer after the headline prompt: 16 steps replayed from a CUDA graph
        _case("decode_7b", "decode", "7b", 1, 4096, steps=16, graph=True),
        # one user's answer on a grouped-query layer, every step a call of its own
        _case("decode_chat_gqa", "decode", "gqa", 1, 2777, steps=8),
        # serving: 32 sequences of very different cache lengths (1024 slabs, 2.4 GB read per step)
        _case("decode_ragged", "decode", "7b", 32, 8192, keep=(0.2, 0.9), steps=4),
        # the same batch on a grouped-query layer
        _case("decode_ragged_gqa", "decode", "gqa", 32, 8192, keep=(0.2, 0.9), steps=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges."""
    kind = rng.choice(["layer", "layer", "layer", "chain", "attend", "decode", "decode", "decode"])
    lo = rng.choice([0.1, 0.2, 0.3, 0.4])
    keep = (lo, min(0.9, lo + rng.choice([0.1, 0.3, 0.5])))
    if kind == "layer":
        arch = rng.choice(["7b", "7b", "gqa", "heads64", "f32", "f32_wide"])
        top = {"7b": 16384, "gqa": 16384, "heads64": 8192, "f32": 512, "f32_wide": 1024}[arch]
        seq = _log_int(rng, 48, top)
        batch = rng.randint(1, max(1, min(8, 16384 // seq if arch[:3] != "f32" else 2)))
        gate = rng.choice(["global", "global", "local"]) if arch != "f32" else "global"
        return _case(None, kind, arch, batch, seq, keep, gate=gate, ragged=batch > 1 and rng.random() < 0.5,
                     window=rng.choice([0, 0, 0, 5, 10]), steps=rng.choice([0, 0, 2, 8]))
    if kind == "chain":
        seq = _log_int(rng, 48, 8192)
        batch = rng.randint(1, max(1, min(8, 16384 // seq)))
        return _case(None, kind, rng.choice(["7b", "gqa"]), batch, seq, keep, steps=rng.choice([0, 0, 4]))
    if kind == "attend":
        return _case(None, kind, rng.choice(["7b", "gqa"]), 1, _log_int(rng, 1024, 16384), keep,
                     empty_heads=rng.choice([0, 2, 8]))
    arch = rng.choice(["7b", "7b", "gqa", "gqa", "heads64"])
    batch = _log_int(rng, 1, 32)
    return _case(None, kind, arch, batch, _log_int(rng, 128, 8192), keep, steps=rng.choice([2, 4, 8]),
                 graph=rng.random() < 0.3)


def _shape(case):
    d, h, hk, D, gh, gD, dt = ARCHS[case["arch"]]
    return inputs.LayerShape(case["batch"], case["seq"], d, h, D, gh, gD, dt, kv_heads=0 if hk == h else hk,
                             recent_window=case["window"])


# ------------------------------------------------------------------ inputs
def _gate_scores(shape, case, X, W, lens):
    """The gate's scores of all valid tokens [kv heads, tokens] from torch's float32 operations: used to
    place gamma only."""
    out = []
    for b in range(shape.batch):
        x = X[b, :lens[b]].float()
        if case["gate"] == "local":
            out.append((x @ W["W_lin"].float()).t())
            continue
        n, g, D = x.shape[0], shape.gate_heads, shape.gate_head_dim
        q, k, v = ((x @ W[w].float()).view(n, g, D) for w in ("Wq_g", "Wk_g", "Wv_g"))
        mask = torch.ones(n, n, dtype=torch.bool, device=x.device).triu(1)
        heads = []
        for i in range(g):
            s = (q[:, i] @ k[:, i].t()).mul_(1.0 / math.sqrt(D)).masked_fill_(mask, -math.inf)
            heads.append(torch.softmax(s, dim=1) @ v[:, i])
        out.append((torch.cat(heads, dim=1) @ W["Wo_g"].float()).t())
    return torch.cat(out, dim=1)


def _gamma(scores, keep, tau):
    """Per-head constant that keeps about keep[i] of the tokens, placed in the widest gap between two
    neighbouring scores near that quantile: a float32 rounding of a score moves no flag."""
    v = torch.sort(scores, dim=1).values
    m = v.shape[1]
    w = max(4, m // 100)
    cuts = []
    for i in range(v.shape[0]):
        k = int(round((1.0 - float(keep[i])) * m))
        lo, hi = min(max(k - w, 1), m - 1), max(min(k + w, m), 2)
        j = torch.argmax(v[i, lo:hi] - v[i, lo - 1:hi - 1]) + lo
        cuts.append(0.5 * (v[i, j] + v[i, j - 1]))
    return (math.log(tau / (1.0 - tau)) - torch.stack(cuts)).float().contiguous()


def _keep_rates(case, n, seed):
    return inputs.keep_targets_uniform(n, seed, case["keep_lo"], case["keep_hi"])


def _decode_buffers(st, shape, case, seed):
    steps = case["steps"]
    st["tokens"] = [inputs.decode_inputs(shape, seed, t, "cuda") for t in range(steps)]
    st["o"] = torch.zeros(steps, shape.batch, shape.heads, shape.head_dim, dtype=shape.torch_dtype, device="cuda")
    st["o_step"] = list(st["o"])
    st["ws_decode"] = ag.workspace(st["desc"], ag.AG_CALL_DECODE)


def prepare(case, seed):
    shape = _shape(case)
    st = {"kind": case["kind"], "gate": case["gate"], "shape": shape, "graph": None, "tokens": []}
    {"layer": _prepare_layer, "chain": _prepare_chain, "attend": _prepare_attend,
     "decode": _prepare_decode}[case["kind"]](st, shape, case, int(seed) * 100000)
    return st


def _attention_buffers(st, shape, steps):
    B, hk, n = shape.batch, shape.kvh, shape.seq
    st["cache"] = ag.RaggedCache.allocate(shape, [n + steps] * (B * hk))
    st["prefix"] = torch.zeros(B, hk, n + 1, dtype=torch.int32, device="cuda")
    st["idx"] = torch.zeros(B, hk, n, dtype=torch.int32, device="cuda")
    st["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    st["O"] = torch.zeros(B, shape.heads, n, shape.head_dim, dtype=shape.torch_dtype, device="cuda")
    st["ws_prefill"] = ag.workspace(st["desc"], ag.AG_CALL_PREFILL)


def _cache_outputs(st):
    c = st["cache"]
    out = [c.len, c.k_rows, c.v_rows, st["status"]]
    if c.pos is not None:
        out += [c.recent_k, c.recent_v, c.recent_live, c.pos]
    return out


def _prepare_layer(st, shape, case, seed):
    B, hk, n = shape.batch, shape.kvh, shape.seq
    lens = np.full(B, n)
    if case["ragged"]:
        lens[1:] = np.random.default_rng(n).integers(max(1, n // 4), n + 1, size=B - 1)
        st["seq_lens"] = torch.tensor(lens, dtype=torch.int32, device="cuda")
    st["desc"] = ag.make_desc(shape, st.get("seq_lens"))
    X = st["X"] = inputs.hidden_states(shape, seed, "cuda")
    W = st["W"] = inputs.layer_weights(shape, seed + 10, "cuda")
    st["Q"], st["K"], st["V"] = inputs.project_qkv(shape, X, W)
    if case["gate"] == "local":
        W["W_lin"] = inputs.linear_gate_weight(shape.with_(heads=hk), seed + 30, "cuda")
    else:
        st["ws_gate"] = ag.workspace(st["desc"], ag.AG_CALL_GATE)
    st["gamma"] = _gamma(_gate_scores(shape, case, X, W, lens), _keep_rates(case, hk, seed), shape.tau)
    st["scores"] = torch.zeros(B, hk, n, dtype=torch.float32, device="cuda")
    st["flags"] = torch.zeros(B, hk, n, dtype=torch.uint8, device="cuda")
    _attention_buffers(st, shape, case["steps"])
    _decode_buffers(st, shape, case, seed + 50)
    # scores and attention outputs at padding positions are unspecified: the sequences themselves come out
    per_seq = [t[b, :, :lens[b]] for t in (st["scores"], st["O"]) for b in range(B)] if case["ragged"] else \
        [st["scores"], st["O"]]
    st["out"] = per_seq + [st["flags"], st["prefix"], st["idx"], st["o"]] + _cache_outputs(st)


def _prepare_chain(st, shape, case, seed):
    X = st["X"] = inputs.hidden_states(shape, seed, "cuda")
    W = st["W"] = inputs.layer_weights(shape, seed + 10, "cuda")
    W["Wo"] = inputs.output_weight(shape, seed + 30, "cuda", n_layers=32)
    st["gamma"] = _gamma(_gate_scores(shape, case, X, W, [shape.seq] * shape.batch),
                         _keep_rates(case, shape.kvh, seed), shape.tau)
    buf = st["buf"] = schedule.ChainedLayerBuffers(ag, shape, case["steps"])
    for t in (buf.scores, buf.flags, buf.prefix, buf.Q, buf.K, buf.V, buf.O):
        t.zero_()
    st["desc"], st["cache"], st["status"] = buf.desc, buf.cache, buf.status
    st["X_next"] = torch.zeros_like(X)
    _decode_buffers(st, shape, case, seed + 50)
    st["out"] = [st["X_next"], buf.scores, buf.flags, buf.prefix, buf.Q, buf.K, buf.V, buf.O, st["o"]] + \
        _cache_outputs(st)


def _prepare_attend(st, shape, case, seed):
    st["desc"] = ag.make_desc(shape)
    hk = shape.kvh
    st["Q"], st["K"], st["V"] = inputs.qkv_gaussian(shape, seed, "cuda")
    keep = _keep_rates(case, hk, seed)
    # heads that keep nothing, at the same share of the key/value heads
    keep[np.random.default_rng(seed).permutation(hk)[:case["empty_heads"] * hk // shape.heads]] = 0.0
    u = torch.rand(shape.batch, hk, shape.seq, device="cuda", generator=torch.Generator("cuda").manual_seed(seed + 5))
    st["flags"] = (u < torch.tensor(keep, dtype=torch.float32, device="cuda")[None, :, None]).to(torch.uint8)
    _attention_buffers(st, shape, 0)
    st["out"] = [st["O"], st["prefix"], st["idx"]] + _cache_outputs(st)


def _prepare_decode(st, shape, case, seed):
    desc = st["desc"] = ag.make_desc(shape)
    L = inputs.ragged_lengths(shape.batch * shape.kvh, shape.seq, seed, case["keep_lo"], case["keep_hi"])
    cap = L + case["steps"]
    off, _ = inputs.slab_layout(cap)
    # a pool sized for the longest caches the batch could have had; the slabs lie tightly in its front
    pool = cap.size * (math.floor(case["keep_hi"] * shape.seq) + case["steps"])
    k, v = (inputs.randn((pool, shape.head_dim), seed + i, "cuda", shape.torch_dtype) for i in (1, 2))
    st["cache"] = ag.RaggedCache(k, v, torch.from_numpy(off).cuda(), torch.from_numpy(cap).cuda(),
                                 torch.from_numpy(L).cuda(), int(cap.max()))
    st["len_prompt"] = st["cache"].len.clone()
    st["status"] = torch.zeros(1, dtype=torch.int32, device="cuda")
    _decode_buffers(st, shape, case, seed + 50)
    st["out"] = [st["o"]] + _cache_outputs(st)
    if case["graph"]:
        side = torch.cuda.Stream()
        side.wait_stream(torch.cuda.current_stream())
        with torch.cuda.stream(side):
            _decode_pass(st)
        torch.cuda.current_stream().wait_stream(side)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            _decode_pass(st)
        st["graph"] = g


# -------------------------------------------------------------------- one pass
def _decode_steps(st):
    desc, cache, status, ws = st["desc"], st["cache"], st["status"], st["ws_decode"]
    for (q, k, v, f), o in zip(st["tokens"], st["o_step"]):
        ag.ag_decode_step(desc, q, k, v, f, cache, 0.0, o, status, ws)


def _decode_pass(st):
    st["cache"].len.copy_(st["len_prompt"])
    _decode_steps(st)


def run(st):
    if st["kind"] == "decode":
        if st["graph"] is not None:
            st["graph"].replay()
        else:
            _decode_pass(st)
        return st["out"]
    if st["kind"] == "chain":
        schedule.chained_layer(ag, st["buf"], st["X"], st["W"], st["gamma"], st["X_next"])
    else:
        desc, W = st["desc"], st.get("W")
        if st["kind"] == "layer":
            if st["gate"] == "local":
                ag.ag_gate_linear_forward(desc, st["X"], W["W_lin"], st["gamma"], st["scores"], st["flags"])
            else:
                ag.ag_gate_forward(desc, st["X"], W["Wq_g"], W["Wk_g"], W["Wv_g"], W["Wo_g"], st["gamma"],
                                   st["scores"], st["flags"], st["ws_gate"])
        ag.ag_compact_kv(desc, st["K"], st["V"], st["flags"], st["cache"], st["prefix"], st["idx"], st["status"], None)
        ag.ag_prefill_attn(desc, st["Q"], st["K"], st["V"], st["flags"], st["cache"], st["prefix"], 0.0, st["O"],
                           st["ws_prefill"])
    if st["tokens"]:
        _decode_steps(st)
    return st["out"]


# ---------------------------------------------------------- work and tolerance
def work(case):
    """Bytes every input is read and every output written once, and the multiply-adds the method needs:
    attention over retained keys only."""
    s = _shape(case)
    B, n, d, h, hk, D, GD = s.batch, s.seq, s.hidden, s.heads, s.kvh, s.head_dim, s.gate_heads * s.gate_head_dim
    e = 4 if s.dtype == "f32" else 2
    keep = 0.5 * (case["keep_lo"] + case["keep_hi"]) * (1.0 - case["empty_heads"] / h)
    row = D * e
    # tokens and token pairs; padded batches: the first sequence is full, the others uniform in [n/4, n]
    tok, pairs = B * n, B * n * (n + 1) / 2
    if case["ragged"]:
        tok, pairs = n * (1 + 0.625 * (B - 1)), (1 + 0.4375 * (B - 1)) * n * (n + 1) / 2
    cached = keep * hk * (B * n if case["kind"] == "decode" else tok)     # rows of K (and of V) in the cache
    byt = flops = 0.0
    if case["kind"] != "decode":
        byt += tok * (2 * h + 2 * hk) * row + 2 * cached * row            # Q, O, K, V; cache rows
        byt += hk * tok * (1 + 4 + (4 if case["kind"] != "chain" else 0))  # flags, prefix, idx
        flops += 4.0 * D * h * (tok + keep * pairs)
    if case["kind"] in ("layer", "chain"):
        byt += tok * d * e + hk * tok * 4                                 # X, scores
        if case["gate"] == "local":
            byt += d * hk * e
            flops += 2.0 * tok * d * hk
        else:
            byt += (3 * d * GD + GD * hk) * e
            flops += 2.0 * tok * d * 3 * GD + 4.0 * GD * pairs + 2.0 * tok * GD * hk
    if case["kind"] == "chain":
        byt += (d * (h + 2 * hk) * D + h * D * d) * e + tok * d * e
        flops += 2.0 * tok * d * (h + 2 * hk) * D + 2.0 * tok * h * D * d
    steps = case["steps"]
    byt += steps * (2 * cached * row + B * (2 * h + 2 * hk) * row)
    flops += steps * 4.0 * D * (h // hk) * cached
    return {"bytes": byt, "flops": flops}


def tolerance(case):
    if ARCHS[case["arch"]][-1] == "f32":
        return {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    return {"rel": 1e-2, "max": 0.2, "differ": 1e-3}
