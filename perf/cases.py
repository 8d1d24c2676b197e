"""The work that a user of this framework has it do, as cases that can be timed.

A serving program prefills a prompt, compresses every layer's K / V into the hybrid cache (fa_compress and its
variants) and then, token by token, pushes a row and attends to the cache (fa_decode_step and its variants).  The
listed cases are those calls at the shapes of the benchmark configurations (a toy fp32 cache, a GQA 4 model at 32K
and 128K tokens, an MHA model at batch 8 and 4K tokens), a short chat, and ragged batches of odd lengths.  ``draw``
gives others between them.

A case:
  op        which public calls a pass makes (see ``run``)
  dtype     storage of K / V / q / out: "bf16" or "f32"
  batch, q_heads, kv_heads, head_dim
  full_k, full_v   dims kept per token; the others are held as n_coef coefficients of period ``period``
  prompt    prefilled tokens (ragged: the longest row)
  l_init, l_local  windows kept whole
  ragged    rows of different length
  layers    caches that a pass works on;  tokens: decode steps per layer that a pass makes
"""
import math
import random

import torch

from paper_2506_11886_b200 import fa, synth

DECODE_OPS = ("step", "step_layers", "append_decode", "step_host")
COMPRESS_OPS = ("compress", "compress_layers", "compress_ragged")
# what compression writes and a step goes on from
BUFFERS = ("k_init", "v_init", "k_local", "v_local", "k_mid", "v_mid", "coef_k", "coef_v", "state")


def _case(op, batch, q_heads, kv_heads, prompt, n_coef, period, l_local, full_k=32, full_v=32, head_dim=128, l_init=4,
          dtype="bf16", ragged=False, layers=1, tokens=0, name=None):
    c = dict(op=op, dtype=dtype, batch=batch, q_heads=q_heads, kv_heads=kv_heads, head_dim=head_dim, full_k=full_k,
             full_v=full_v, n_coef=n_coef, period=period, prompt=prompt, l_init=l_init, l_local=l_local, ragged=ragged,
             layers=layers, tokens=tokens)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a toy fp32 cache is built and asked once (benchmark configuration 0)
        _case("request", 1, 4, 1, 1024, 64, 1024, 0, l_init=0, dtype="f32", tokens=1, name="toy_f32_request"),
        # a short chat, one user: a model's forward pass calls the step layer by layer
        _case("step", 1, 32, 8, 2048, 256, 4096, 1024, layers=7, tokens=2, name="decode_2k_chat"),
        # the headline: one user at 32K tokens, all layers of a token enqueued by one call
        _case("step_layers", 1, 32, 8, 32000, 1024, 32768, 1024, layers=4, tokens=4, name="decode_32k"),
        # the same with the token's q, k, v and result in pinned host memory, the result awaited every step
        _case("step_host", 1, 32, 8, 32000, 1024, 32768, 1024, tokens=8, name="decode_host_32k"),
        # MHA serving, batch 8
        _case("step_layers", 8, 32, 32, 4000, 256, 4096, 1024, 48, 48, layers=4, tokens=2, name="decode_4k_mha_b8"),
        # long context, batch 4
        _case("step_layers", 4, 32, 8, 131000, 2048, 131072, 2048, layers=2, tokens=2, name="decode_128k_b4"),
        # a batch of users at different places, three query heads to a KV head, kept dims that differ for K and V;
        # the program pushes and attends by separate calls
        _case("append_decode", 6, 24, 8, 12345, 512, 16384, 1024, 24, 40, ragged=True, layers=2, tokens=2, name="decode_ragged_b6"),
        # prefill compression of a stage of layers in one call
        _case("compress_layers", 1, 32, 8, 32768, 1024, 32768, 1024, layers=6, name="compress_32k_layers"),
        # prefill compression of one layer: MHA serving batch; the longest prompt; a ragged batch of odd lengths
        _case("compress", 8, 32, 32, 4096, 256, 4096, 1024, 48, 48, name="compress_4k_mha_b8"),
        _case("compress", 4, 32, 8, 131072, 2048, 131072, 2048, name="compress_128k_b4"),
        _case("compress_ragged", 6, 24, 8, 12345, 512, 16384, 1024, 24, 40, ragged=True, name="compress_ragged_b6"),
        # offline calibration: which dims to keep
        _case("select", 1, 32, 8, 32768, 1024, 32768, 1024, name="select_32k"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(("request", "step", "step_layers", "step_layers", "append_decode", "step_host", "compress",
                     "compress_layers", "compress_ragged", "select"))
    f32 = op == "request"
    q_heads, kv_heads, d = rng.choice(((4, 1, 128), (8, 2, 64), (8, 2, 128)) if f32 else ((32, 8, 128), (32, 8, 128), (24, 8, 128), (32, 32, 128), (16, 4, 64)))
    batch = 1 if op in ("select", "step_host") else _log_int(rng, 1, 8)
    ragged = op == "compress_ragged" or (op == "append_decode" and rng.random() < 0.5)
    # the prefilled tensors of a layer stay at or below those of the longest listed prompt
    longest = min(131072, (1 << 29) // (batch * kv_heads * d))
    if op in ("select", "compress_layers"):
        longest = min(longest, 32768)
    prompt = _log_int(rng, 500, 2000 if f32 else longest)
    if f32:
        l_init, l_local = rng.choice(((0, 0), (4, 64), (4, 256)))
    else:
        l_init, l_local = 4, 2048 if prompt > 65536 else 1024 if prompt > 1500 else 256
    period = 1 << max(10, (prompt + 16 - 1).bit_length())          # room for the tokens to come
    n_coef = min(2048, max(64, period // rng.choice((16, 32, 64))))
    full = (16, 24, 32, 40, 48, 64) if d == 128 else (8, 16, 24, 32)
    layers = rng.randint(1, 4) if op in ("step", "step_layers", "append_decode", "compress_layers") else 1
    tokens = 1 if f32 else rng.randint(1, 4) if op in DECODE_OPS else 0
    while layers > 1 and layers * batch * prompt * kv_heads * d > 1 << 29:
        layers -= 1
    return _case(op, batch, q_heads, kv_heads, prompt, n_coef, period, l_local, rng.choice(full), rng.choice(full), d, l_init,
                 "f32" if f32 else "bf16", ragged, layers, tokens)


def _shape(c):
    return synth.Shape(c["op"], B=c["batch"], layers=c["layers"], Hq=c["q_heads"], Hkv=c["kv_heads"], d=c["head_dim"],
                       L=c["prompt"], dtype=c["dtype"], n_full_k=c["full_k"], n_full_v=c["full_v"], M=c["n_coef"],
                       T=c["period"], L_init=c["l_init"], L_local=c["l_local"])


def _layout(c):
    # one residue class of the middle per transform of n_coef / 2 points, as the benchmark lays its caches out
    return fa.Layout(batch=c["batch"], n_q_heads=c["q_heads"], n_kv_heads=c["kv_heads"], head_dim=c["head_dim"],
                     n_full_k=c["full_k"], n_full_v=c["full_v"], n_coef=c["n_coef"], period=c["period"],
                     l_init=c["l_init"], l_local=c["l_local"], max_mid=c["period"],
                     mid_classes=2 * c["period"] // c["n_coef"],
                     kv_dtype=fa.FA_F32 if c["dtype"] == "f32" else fa.FA_BF16)


def _lengths(c, seed=None):
    """Tokens of every batch row (without a seed: what they are on average)."""
    if not c["ragged"]:
        return [c["prompt"]] * c["batch"]
    if seed is None:
        return [0.6 * c["prompt"]] * c["batch"]
    rng = random.Random(seed * 7919 + 11)
    # the longest row is there; with the other rows' sum held, every seed is about the same work
    part = [0.52 + (i - (c["batch"] - 2) / 2) * 0.7 / max(1, c["batch"] - 1) for i in range(c["batch"] - 1)]
    rows = [max(1, min(c["prompt"], int(c["prompt"] * p) + rng.randint(-40, 40))) for p in part] + [c["prompt"]]
    rng.shuffle(rows)
    return rows


def prepare(case, seed):
    c, op = case, case["op"]
    shape, layout = _shape(c), _layout(c)
    s = {"case": c, "layout": layout, "lengths": _lengths(c, seed)}
    streams = [synth.KVStream(shape, seed=seed, layer=i, device="cuda", freq="offgrid") for i in range(c["layers"])]
    if op == "select":
        s["K"], s["V"] = ([t] for t in streams[0].tokens(0, c["prompt"], work_dtype=torch.float32))
        return s
    s["caches"] = [fa.Cache(layout, st.idx_full_k, st.idx_full_v) for st in streams]
    s["ws"] = fa.new_workspace(layout)
    if op in COMPRESS_OPS or op == "request":
        prefill = [st.tokens(0, c["prompt"], work_dtype=torch.float32) for st in streams]
        s["K"], s["V"] = [p[0] for p in prefill], [p[1] for p in prefill]
        if op == "request":
            s["q"] = synth.queries(shape, seed=seed, device="cuda")
            s["out"] = torch.zeros_like(s["q"])
        return s
    n = c["tokens"]
    q, k, v = [], [], []
    for i, (st, cache) in enumerate(zip(streams, s["caches"])):
        K, V = st.tokens(0, c["prompt"], work_dtype=torch.float32)
        if c["ragged"]:
            fa.fa_compress_ragged(layout, cache, K, V, s["lengths"], s["ws"])
        else:
            fa.fa_compress(layout, cache, K, V, s["ws"])
        del K, V
        q.append(torch.stack([synth.queries(shape, seed=seed, step=t, layer=i, device="cuda") for t in range(n)]))
        K, V = st.tokens(c["prompt"], c["prompt"] + n, work_dtype=torch.float32)
        k.append(K.transpose(0, 1).contiguous())
        v.append(V.transpose(0, 1).contiguous())
    # [token][layer][batch][head][dim]
    q, k, v = (torch.stack(x, dim=1).contiguous() for x in (q, k, v))
    out = torch.zeros_like(q)
    s["at_prompt"] = [cache.state.clone() for cache in s["caches"]]
    if op == "step_layers":
        s["args"] = [fa.LayerStep([layout] * c["layers"], s["caches"], list(q[t]), list(k[t]), list(v[t]), list(out[t])) for t in range(n)]
    if op == "step_host":
        q, k, v = (x.cpu().pin_memory() for x in (q, k, v))
        out = torch.zeros(q.shape, dtype=q.dtype).pin_memory()
        s["staging"] = torch.zeros(fa.fa_step_staging_bytes(layout), dtype=torch.uint8, device="cuda")
    s["q"], s["k"], s["v"], s["out"] = q, k, v, out
    s["views"] = [[tuple(x[t][i] for x in (q, k, v, out)) for i in range(c["layers"])] for t in range(n)]
    return s


def _updated(s):
    return [{n: getattr(cache, n) for n in BUFFERS} for cache in s["caches"]]


def run(state):
    s, layout = state, state["layout"]
    c = s["case"]
    op = c["op"]
    if op == "select":
        return fa.fa_select_dims(layout, s["K"][0], s["V"][0])
    caches, ws = s["caches"], s["ws"]
    if op == "request":
        fa.fa_compress(layout, caches[0], s["K"][0], s["V"][0], ws)
        fa.fa_decode_attention(layout, caches[0], s["q"], s["out"], ws)
        return {"out": s["out"], "caches": _updated(s)}
    if op == "compress":
        fa.fa_compress(layout, caches[0], s["K"][0], s["V"][0], ws)
        return _updated(s)
    if op == "compress_ragged":
        fa.fa_compress_ragged(layout, caches[0], s["K"][0], s["V"][0], s["lengths"], ws)
        return _updated(s)
    if op == "compress_layers":
        fa.fa_compress_layers([layout] * len(caches), caches, s["K"], s["V"], ws)
        return _updated(s)
    # A generation: the counters go back to where the prompt ended (as when a program tries several continuations),
    # so that the middle has room however often a pass is made; then c["tokens"] steps.
    for cache, at in zip(caches, s["at_prompt"]):
        cache.state.copy_(at)
    for t in range(c["tokens"]):
        if op == "step_layers":
            fa.fa_decode_step_layers(s["args"][t], ws)
            continue
        for cache, (q, k, v, out) in zip(caches, s["views"][t]):
            if op == "step":
                fa.fa_decode_step(layout, cache, q, k, v, out, ws)
            elif op == "append_decode":
                fa.fa_append(layout, cache, k, v)
                fa.fa_decode_attention(layout, cache, q, out, ws)
            else:
                fa.fa_decode_step_host(layout, cache, q, k, v, out, s["staging"], ws)
                torch.cuda.current_stream().synchronize()           # the program reads out before it goes on
    return {"out": s["out"], "caches": _updated(s)}


def work(case):
    c = case
    eb = 2 if c["dtype"] == "bf16" else 4
    d, M, G = c["head_dim"], c["n_coef"], c["q_heads"] // c["kv_heads"]
    comp = 2 * d - c["full_k"] - c["full_v"]                         # compressed dims of K and V
    kept = c["full_k"] + c["full_v"]
    heads = c["kv_heads"] * c["layers"]
    byts = flops = 0.0
    for L in _lengths(c):
        win = min(L, c["l_init"] + c["l_local"])
        mid = L - win
        rows = (mid * kept + win * 2 * d) * eb                       # K^mu, V^mu and the windows
        coef = M * comp * 4
        if c["op"] in COMPRESS_OPS or c["op"] in ("request", "select"):
            # the prefill in, the cache out; the projection on the basis as Eq.3 states it
            byts += heads * L * 2 * d * eb
            byts += c["kv_heads"] * 2 * d * 8 if c["op"] == "select" else heads * (rows + coef)
            flops += heads * 2 * M * mid * (2 * 2 * d if c["op"] == "select" else comp)  # select projects and rebuilds every dim
        if c["op"] in DECODE_OPS or c["op"] == "request":
            n = c["tokens"]
            # the cache in; a push reads and writes every coefficient (the read serves the query too)
            byts += n * heads * (rows + coef * (1 if c["op"] == "request" else 2) + (2 * G + 4) * d * eb)
            # products with the kept dims, with the coefficients, and the transforms between bins and tokens
            flops += n * heads * G * (4 * d * win + 2 * kept * mid + 2 * M * comp + 5 * mid * math.log2(M))
    return {"bytes": byts, "flops": flops}


def tolerance(case):
    if case["dtype"] == "f32":
        return {"rel": 2e-5, "max": 2e-3}
    if case["op"] in COMPRESS_OPS:
        # fp32 sums of bf16 inputs over a basis rounded to bf16; single coefficients far below the spectrum's peaks carry the peaks' rounding
        return {"rel": 2e-3, "max": 0.1}
    if case["op"] == "select":
        return {"rel": 5e-3, "max": 0.1}
    return {"rel": 1e-2, "max": 0.2}                                 # bf16 results
