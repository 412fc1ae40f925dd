"""The work this library is used for, as cases that can be timed and compared: sink prediction, bulk and chunked appends,
decode steps and prompt attention, through the public Python entry points.

A case is one kind of call over one layer's cache:
  predict  sink prediction over a prompt's hidden state at the emergence layer
  append   quantization of a prompt, or of a chunk of one, into the cache
  decode   one decode step of a layer: append the new token, attend over the cache
  prompt   a prompt (or a chunk of one) through a layer: append it, then attend with all of its queries
Shapes are those of paper_2508_04257_b200/synth.py (LLaMA2-7B- and LLaMA3-8B-shaped layers, the 32-layer decode batch, the
long-context layer, the small 64-channel-head layer) and shapes between them.  Values have the structure synth.py gives
them: a few sink tokens with extreme hidden channels and small-norm K and V, keys with loud channels off zero, queries half
of which look at a sink key.  Every pass starts from the same cache length, so it can be repeated on the same state: chunks
either start on a group boundary or end on one, which leaves the open group's earlier rows untouched.
"""
import math

import torch

import paper_2508_04257_b200 as kv

PFN = 1                     # Preserve-First-N beside the predicted tokens
NARROW = 64                 # hidden width where the hidden state is only there to place the sinks
NARROW_CHANNELS = (5, 9)


def _layer(kind, name, batch, hq, hkv, dim, bits, group, start, tokens, topk, scheme="dynamic"):
    return {"name": name, "kind": kind, "batch": batch, "hq": hq, "hkv": hkv, "dim": dim, "bits": bits, "group": group,
            "start": start, "tokens": tokens, "topk": topk, "scheme": scheme}


def listed():
    return [
        # sink prediction for a batch of LLaMA2-7B prompts: two outlier channels, once per prompt
        {"name": "predict_7b", "kind": "predict", "batch": 8, "seq": 4096, "hidden": 4096, "channels": 2, "topk": 8},
        # prompt of a LLaMA2-7B-shaped layer, 2 bit
        _layer("append", "append_prompt_2bit", 8, 32, 32, 128, 2, 128, 0, 4096, 8),
        # prompts of a large decode batch, 4 bit, 64-token groups
        _layer("append", "append_batch_4bit", 16, 32, 32, 128, 4, 64, 0, 8192, 16),
        # the last chunk of a chunked prefill, 3 bit: starts inside an open group, ends on a boundary
        _layer("append", "append_chunk_3bit", 5, 32, 8, 128, 3, 64, 3237, 2779, 11),
        # one interactive sequence of the small 64-channel-head layer: latency
        _layer("decode", "decode_small_4bit", 1, 8, 8, 64, 4, 32, 256, 1, 2),
        # decode step of a LLaMA2-7B-shaped layer, 2 bit
        _layer("decode", "decode_layer_2bit", 8, 32, 32, 128, 2, 128, 4096, 1, 8),
        # the same layer with calibrated parameters (the paper's main comparison), ragged length
        _layer("decode", "decode_static_2bit", 8, 32, 32, 128, 2, 128, 3821, 1, 8, "static"),
        # one long context with grouped queries and 1 % sink tokens
        _layer("decode", "decode_long_gqa_2bit", 1, 32, 8, 128, 2, 128, 131072, 1, 1311),
        # a middle-sized decode batch, 3 bit, a length inside a group
        _layer("decode", "decode_batch_3bit", 16, 32, 32, 128, 3, 64, 8101, 1, 16),
        # the large decode batch, 4 bit
        _layer("decode", "decode_batch_4bit", 64, 32, 32, 128, 4, 64, 8192, 1, 16),
        # whole prompts of a LLaMA2-7B-shaped layer, 2 bit
        _layer("prompt", "prompt_layer_2bit", 8, 32, 32, 128, 2, 128, 0, 4096, 8),
        # a ragged chunk of a long prompt with grouped queries, 4 bit
        _layer("prompt", "prompt_chunk_gqa_4bit", 1, 32, 8, 128, 4, 64, 6400, 1003, 33),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["predict", "append", "append", "decode", "decode", "decode", "prompt", "prompt"])
    if kind == "predict":
        seq, hidden = _log_int(rng, 128, 131072), rng.choice([512, 2048, 4096])
        batch = max(1, min(_log_int(rng, 1, 64), (1 << 28) // (seq * hidden)))
        return {"kind": kind, "batch": batch, "seq": seq, "hidden": hidden, "channels": rng.choice([1, 2, 2, 3, 4]),
                "topk": max(1, min(seq, rng.choice([2, 8, 16, seq // 100])))}
    hkv = rng.choice([4, 8, 8, 32])
    hq = hkv * rng.choice([1, 1, 4, 4, 2, 8]) if hkv < 32 else 32
    bits, group, dim = rng.choice([2, 3, 4]), rng.choice([32, 64, 64, 128, 128]), 128
    if rng.random() < 0.1:
        bits, group, dim = rng.choice([2, 4]), rng.choice([32, 64]), 64
    scheme = "dynamic"
    if kind in ("append", "decode") and dim == 128 and rng.random() < 0.3:
        scheme = rng.choice(["static", "per_token"])
        group = rng.choice([64, 128])          # one or two channel groups per row
        if scheme == "per_token":
            hq = hkv
            group = 128 if bits == 3 else group
    # cached elements of K: up to those of the large decode batch (appends: a quarter of it; prompts also by their pairs)
    limit = {"decode": 1 << 31, "append": 1 << 29, "prompt": 1 << 27}[kind]
    seq = _log_int(rng, 64, 131072 if kind == "decode" else 16384 if kind == "append" else 8192)
    batch = max(1, min(_log_int(rng, 1, 64), limit // (seq * hkv * dim)))
    if kind == "prompt":
        batch = max(1, min(batch, (1 << 32) // (seq * seq * hq)))
    if kind == "decode":
        start, tokens = seq, 1
    elif rng.random() < 0.5:                   # a whole prompt, or a chunk that starts on a group boundary
        start = rng.choice([0, seq // 2 // group * group])
        tokens = max(2, seq - start)
    else:                                      # a chunk that ends on one
        end = max(2 * group, seq // group * group)
        start = rng.randrange(end // 4, end - 1)
        tokens = end - start
    topk = min(rng.choice([2, 8, 16, max(1, seq // 100)]), seq)
    case = _layer(kind, "", batch, hq, hkv, dim, bits, group, start, tokens, topk, scheme)
    del case["name"]
    return case


def _gen(seed):
    g = torch.Generator("cuda")
    g.manual_seed(int(seed))
    return g


def _plant(batch, seq, topk, hidden, channels, g):
    """Hidden state with outliers on `channels` at token 0 and topk - 1 others; beyond 64 sinks they come in runs of 16."""
    k = min(topk, seq)
    H = torch.randn((batch, seq, hidden), device="cuda", generator=g, dtype=torch.float16)
    run = 16 if k > 64 else 1
    order = torch.rand((batch, -(-seq // run)), device="cuda", generator=g)
    order[:, 0] = 2.0
    first = order.topk(min(-(-k // run), order.shape[1]), dim=1).indices * run
    pos = (first[:, :, None] + torch.arange(run, device="cuda")).reshape(batch, -1).clamp_(max=seq - 1)[:, :k]
    rows = torch.arange(batch, device="cuda")[:, None]
    for c in channels:
        size = 1000.0 * (1.0 + 0.25 * torch.rand(pos.shape, device="cuda", generator=g))
        sign = torch.where(torch.rand(pos.shape, device="cuda", generator=g) < 0.5, -1.0, 1.0)
        H[rows, pos, c] = (size * sign).half()
    return H, pos


def _keys_values(case, tokens, pos, g):
    """K, V [B, Hkv, tokens, D]: four loud channels off zero per head in K; small-norm rows at the sink positions `pos`."""
    B, h, d = case["batch"], case["hkv"], case["dim"]
    K = torch.randn((B, h, tokens, d), device="cuda", generator=g, dtype=torch.float16)
    V = torch.randn((B, h, tokens, d), device="cuda", generator=g, dtype=torch.float16)
    gain, off = torch.ones((h, d), device="cuda"), torch.zeros((h, d), device="cuda")
    loud = torch.rand((h, d), device="cuda", generator=g).topk(4, dim=1).indices
    gain.scatter_(1, loud, 20.0)
    shift = 4.0 + 8.0 * torch.rand(loud.shape, device="cuda", generator=g)
    off.scatter_(1, loud, torch.where(torch.rand(loud.shape, device="cuda", generator=g) < 0.5, -shift, shift))
    K.mul_(gain[:, None].half()).add_(off[:, None].half())
    if pos is not None:
        at = pos[:, None, :, None].expand(B, h, pos.shape[1], d)
        for x in (K, V):
            x.scatter_(2, at, x.gather(2, at) * 0.02)
    return K, V


def _queries(case, tokens, sink_key, g):
    """[B, Hq, tokens, D]: N(0,1); every other head pulled four units toward a sink key of its KV head."""
    B, hq, d, rep = case["batch"], case["hq"], case["dim"], case["hq"] // case["hkv"]
    q = torch.randn((B, hq, tokens, d), device="cuda", generator=g, dtype=torch.float16)
    k = sink_key.float()
    k = 4.0 * k / k.norm(dim=-1, keepdim=True).clamp_min(1e-6)
    q[:, ::2] += k.repeat_interleave(rep, dim=1)[:, ::2, None].half()
    return q


class _State:
    pass


def prepare(case, seed):
    g, s = _gen(seed), _State()
    s.kind = case["kind"]
    if s.kind == "predict":
        B, S, d = case["batch"], case["seq"], case["hidden"]
        channels = tuple(range(37, d, d // case["channels"]))[: case["channels"]]
        s.cfg = kv.Config(B, 32, 32, 128, d, 2, 128, -(-S // 128) * 128, case["topk"], PFN, channels)
        s.hidden, _ = _plant(B, S, case["topk"], d, channels, g)
        s.sinks = kv.SinkSet(s.cfg)
        return s
    group, start, tokens = case["group"], case["start"], case["tokens"]
    total = start + tokens
    prompt = start if s.kind == "decode" else total              # tokens the sinks were predicted from
    s.scheme, s.start = case["scheme"], start
    s.cfg = kv.Config(case["batch"], case["hq"], case["hkv"], case["dim"], NARROW, case["bits"], group, (total // group + 1) * group,
                      case["topk"], PFN, NARROW_CHANNELS)
    hidden, pos = _plant(case["batch"], prompt, case["topk"], NARROW, NARROW_CHANNELS, g)
    sinks = kv.predict_sinks(s.cfg, hidden, kv.SinkSet(s.cfg))
    del hidden
    K, V = _keys_values(case, prompt, pos, g)
    s.cache = kv.KVCache(s.cfg, sinks, per_token_keys=s.scheme == "per_token")
    s.params = kv.calibrate(s.cfg, K, V, sinks) if s.scheme == "static" else None
    if start:
        _append(s, K[:, :, :start], V[:, :, :start])
    if s.kind == "decode":
        s.k, s.v = _keys_values(case, 1, None, g)
        s.q = _queries(case, 1, K[:, :, 0], g)[:, :, 0].contiguous()
    else:
        s.k, s.v = (x[:, :, start:].contiguous() for x in (K, V)) if start else (K, V)
        if s.kind == "prompt":
            s.q = _queries(case, tokens, K[:, :, 0], g)
    return s


def _append(s, k, v):
    if s.scheme == "static":
        kv.quantize_append_calibrated(s.cfg, s.cache, s.params, k, v)
    elif s.scheme == "per_token":
        kv.quantize_append_pertoken(s.cfg, s.cache, k, v)
    else:
        kv.quantize_append(s.cfg, s.cache, k, v)


def run(s):
    if s.kind == "predict":
        kv.predict_sinks(s.cfg, s.hidden, s.sinks)
        return [s.sinks.bitmask, s.sinks.pos, s.sinks.count]
    c = s.cache
    c.seq_len = s.start                                          # the pass starts over from the cached prefix
    _append(s, s.k, s.v)
    state = [c.k_codes, c.v_codes, c.k_scale, c.k_zero, c.v_scale, c.v_zero, c.k_tail, c.sink_k, c.sink_v]
    if s.kind == "append":
        return state
    if s.kind == "prompt":
        return list(kv.prefill_attention(s.cfg, c, s.q, s.start)) + state
    if s.scheme == "static":
        out, lse = kv.decode_attention_calibrated(s.cfg, c, s.params, s.q)
    elif s.scheme == "per_token":
        out, lse = kv.decode_attention_pertoken(s.cfg, c, s.q)
    else:
        out, lse = kv.decode_attention(s.cfg, c, s.q)
    return [out, lse] + state


def work(case):
    if case["kind"] == "predict":
        # one 32-byte sector per token and listed channel (the outlier channels lie far apart), mask and positions
        B, S = case["batch"], case["seq"]
        return {"bytes": B * (S * case["channels"] * 32 + S / 8 + 4 * (case["topk"] + PFN)), "flops": 0}
    B, hq, hkv, d, bits, group = (case[k] for k in ("batch", "hq", "hkv", "dim", "bits", "group"))
    start, T, ngv = case["start"], case["tokens"], d // min(group, d)
    params = {"dynamic": 8 * d / group + 8 * ngv, "static": 0, "per_token": 16 * ngv}[case["scheme"]]
    coded = 2 * d * bits / 8 + params                            # one token of one KV head in the cache
    append = B * hkv * T * (2 * d * 2 + coded)                   # fp16 K and V read, codes and parameters written
    if case["kind"] == "append":
        return {"bytes": append, "flops": 0}
    rows = B * hq * T * (2 * d + 4 * d + 4)                      # queries read, outputs and lse written
    cached = B * hkv * (start * coded + (case["topk"] + PFN) * 4 * d)
    pairs = B * hq * (T * start + T * (T + 1) / 2)
    return {"bytes": append + rows + cached, "flops": 4 * d * pairs}


def tolerance(case):
    # integers, codes, parameters and moved rows are defined bit by bit
    if case["kind"] in ("predict", "append"):
        return "exact"
    # four times what the attention outputs measured against float64 attention over the same cache (shapes like the listed
    # ones, every code width): decode 9e-5 and 8e-4, prompts 1.9e-4 and 3.2e-3 (3 bit)
    if case["kind"] == "decode":
        return {"rel": 4e-4, "max": 4e-3, "differ": 0.0}
    return {"rel": 8e-4, "max": 1.3e-2, "differ": 0.0}


def _codes(x, scale, zero, qmax):
    """The value a code stands for, in 64 bits: codes by the format's own 32-bit formula."""
    code = (torch.round(x / torch.where(scale == 0, 1.0, scale)) + zero).clamp_(0, qmax)
    return scale.double() * (code.double() - zero.double())


def _pairs(mn, mx, qmax):
    """(scale, zero) of groups with extremes mn, mx (infinite where a group has no member)."""
    r = mx - mn
    scale = torch.where(r == 0, torch.where(mn == 0, 1.0, mn.abs()), r / torch.full_like(r, qmax))   # a tensor: by a number it would be a product with 1 / qmax
    zero = 0.0 - torch.round(mn / scale)
    none = torch.isinf(mn)
    return torch.where(none, 0.0, scale), torch.where(none, 0.0, zero)


def _extremes(x, sink, dims):
    return (x.masked_fill(sink, math.inf).amin(dims, keepdim=True), x.masked_fill(sink, -math.inf).amax(dims, keepdim=True))


def _as_cached(case, K, V, sink, params):
    """One sequence's keys and values [Hkv, n, D] as the cache holds them, in 64 bits; sink [n]."""
    h, n, d = K.shape
    qmax, G = float(2 ** case["bits"] - 1), case["group"]
    gv, keep = min(G, d), sink[None, :, None]
    k, v = K.float(), V.float()
    by_group = lambda x: x.view(h, n, d // gv, gv)
    token_pairs = lambda x: _pairs(*_extremes(by_group(x), keep[..., None], -1), qmax)
    if case["scheme"] == "static":
        kd = _codes(k, params["k"][0][:, None], params["k"][1][:, None], qmax)
        vd = _codes(by_group(v), *(p[:, None, :, None] for p in params["v"]), qmax).view(h, n, d)
    else:
        vd = _codes(by_group(v), *token_pairs(v), qmax).view(h, n, d)
        if case["scheme"] == "per_token":
            kd = _codes(by_group(k), *token_pairs(k), qmax).view(h, n, d)
        else:
            kd, body = k.double(), n // G * G                    # the open group stays as it came
            kg, sg = k[:, :body].view(h, body // G, G, d), sink[:body].view(1, body // G, G, 1)
            kd[:, :body] = _codes(kg, *_pairs(*_extremes(kg, sg, 2), qmax), qmax).view(h, body, d)
    return torch.where(keep, k.double(), kd), torch.where(keep, v.double(), vd)


def exact(case, seed):
    """Attention outputs in 64 bits over the values that the cache's codes, parameters and exact rows stand for."""
    if case["kind"] in ("predict", "append"):
        return None                                              # integers, codes and moved rows: compared bit by bit
    g = _gen(seed)
    B, hq, hkv, d, start, T = (case[k] for k in ("batch", "hq", "hkv", "dim", "start", "tokens"))
    rep, decode = hq // hkv, case["kind"] == "decode"
    prompt = start if decode else start + T
    hidden, pos = _plant(B, prompt, case["topk"], NARROW, NARROW_CHANNELS, g)
    score = hidden[:, :, list(NARROW_CHANNELS)].abs().amax(-1)
    sinks = torch.zeros((B, start + T), dtype=torch.bool, device="cuda")
    sinks.scatter_(1, score.sort(dim=1, descending=True, stable=True).indices[:, : case["topk"]], True)
    sinks[:, :PFN] = True
    del hidden
    K, V = _keys_values(case, prompt, pos, g)
    params = None
    if case["scheme"] == "static":
        ngv, keep = d // min(case["group"], d), sinks[:, None, :prompt, None]
        ext = lambda x, s, dims: [f([e(x[b : b + 1].float(), s[b : b + 1], dims) for b in range(B)])
                                  for e, f in ((lambda *a: _extremes(*a)[0], lambda m: torch.stack(m).amin(0)),
                                               (lambda *a: _extremes(*a)[1], lambda m: torch.stack(m).amax(0)))]
        qmax = float(2 ** case["bits"] - 1)
        params = {"k": [p.view(hkv, d) for p in _pairs(*ext(K, keep, (0, 2)), qmax)],
                  "v": [p.view(hkv, ngv) for p in _pairs(*ext(V.view(B, hkv, prompt, ngv, -1), keep[..., None], (0, 2, 4)), qmax)]}
    if decode:
        k1, v1 = _keys_values(case, 1, None, g)
        q = _queries(case, 1, K[:, :, 0], g)
    else:
        q = _queries(case, T, K[:, :, 0], g)
    out = torch.empty((B, hq, T, d), dtype=torch.float64, device="cuda")
    lse = torch.empty((B, hq, T), dtype=torch.float64, device="cuda")
    seen = torch.arange(start + T, device="cuda")[None] <= start + torch.arange(T, device="cuda")[:, None]
    for b in range(B):
        kb, vb = (torch.cat([K[b], k1[b]], 1), torch.cat([V[b], v1[b]], 1)) if decode else (K[b], V[b])
        for h in range(hkv):
            sub = {n: [p[h : h + 1] for p in x] for n, x in params.items()} if params else None
            kd, vd = _as_cached(case, kb[h : h + 1], vb[h : h + 1], sinks[b], sub)
            for i in range(h * rep, (h + 1) * rep):
                s = (q[b, i].double() @ kd[0].T / math.sqrt(d)).masked_fill_(~seen, -math.inf)
                lse[b, i] = s.logsumexp(-1)
                out[b, i] = (s - lse[b, i][:, None]).exp_() @ vd[0]
    if decode:
        out, lse = out[:, :, 0], lse[:, :, 0]
    return [out, lse] + [None] * 9
