"""Timed cases of the decode engine: what a text-to-speech program has it do, through the public calls.

A case is one session on one engine.  The streams of the session are opened by one prefill call over
their conditioning prefixes, decoded for a number of steps, and released; prefill-only cases stop after
the first token.  The sizes are those of the workloads in ``paper_2607_21042_b200/cases.py`` and of the
ranges around them: 1 to 128 concurrent utterances, prefixes from a few rows to most of the 2048-token
context, weights in bf16 / W8A16 / W4A16, KV cache in bf16 or e4m3, greedy and top-k sampling, device
and host buffers, given and on-device assembled prefixes, and the continuous batcher.

Model.  The architecture of the workloads with random weights (N(0, 0.02), LayerNorm gamma 1 + N(0, 0.01)),
quantized as the boundary formats are.  Purely random weights have nearly tied logits, which a trained
model has not: one token in sixty would depend on the order of a sum.  Token embeddings therefore
have unit variance like the prefix rows, and every row of the LM head points to the embedding of one
token, so that each token has a confident successor (probability about 0.99 with top-k 30).
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_21042_b200 import binding as B
from paper_2607_21042_b200 import cases as C
from paper_2607_21042_b200.batcher import ContinuousBatcher

DEV = "cuda:0"
MAX_CONTEXT = 2048
TEXT_ROWS = 2048            # text region of the merged embedding table (prefill_tokens)
N_COND = 34                 # 32 speaker latents, emotion, speed
WEIGHTS = {"bf16": C.W_BF16, "w8a16": C.W_INT8_PC, "w4a16": C.W_INT4_G128}
KV = {"bf16": C.KV_BF16, "e4m3": C.KV_FP8_E4M3}


def _case(name, call, streams, lo, hi, steps, model="full", weights="bf16", kv="bf16", top_k=0, logits=False, requests=0):
    """call: decode_steps (one call for all steps), decode_step (a call for each step), decode_step_host (a call for
    each step, host buffers), prefill, prefill_tokens, batcher.  Prefix lengths are spread over lo..hi."""
    c = {"call": call, "model": model, "weights": weights, "kv": kv, "streams": streams, "prefix_lo": lo, "prefix_hi": hi,
         "steps": steps, "top_k": top_k, "logits": logits, "requests": requests}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest session: the two-layer configuration, one utterance, one call for each token
        _case("tiny_b1_p64", "decode_step", 1, 64, 64, 32, model="tiny", logits=True),
        # one utterance, the common request: a 400-row prefix, a chunk of about a second of audio
        _case("bf16_b1_p400", "decode_steps", 1, 400, 400, 64, logits=True),
        # interactive use: int8 weights, sampled, every step's token, logits and hidden row read by the host
        _case("w8a16_b1_p400_topk30_host", "decode_step_host", 1, 400, 400, 48, weights="w8a16", top_k=30, logits=True),
        # a few utterances far into a long context (voice prompt and text of a whole paragraph), odd batch
        _case("w4a16_b3_p1500-1900", "decode_steps", 3, 1500, 1900, 48, weights="w4a16"),
        # a small server: sixteen ragged utterances, int4 weights
        _case("w4a16_b16_p200-800", "decode_steps", 16, 200, 800, 48, weights="w4a16", logits=True),
        # an odd batch in the range where many requests share a GPU, int8 weights, sampled
        _case("w8a16_b37_p50-1100_topk30", "decode_steps", 37, 50, 1100, 40, weights="w8a16", top_k=30),
        # a full server: 128 ragged utterances
        _case("bf16_b128_p200-1200", "decode_steps", 128, 200, 1200, 64),
        # the same with the smallest formats: int4 weights, 8-bit KV cache
        _case("w4a16_b128_e4m3_p200-1200", "decode_steps", 128, 200, 1200, 64, weights="w4a16", kv="e4m3"),
        # 8-bit KV cache on a small batch
        _case("bf16_b9_e4m3_p300-1500", "decode_steps", 9, 300, 1500, 48, kv="e4m3"),
        # time to the first token of one utterance, odd length
        _case("prefill_bf16_b1_p777", "prefill", 1, 777, 777, 0, logits=True),
        # time to the first token of a group of requests, prefix assembled on the device from text ids
        _case("prefill_tokens_w8a16_b8_p60-260", "prefill_tokens", 8, 60, 260, 0, weights="w8a16", logits=True),
        # requests arriving at a server of sixteen slots: admission, chunked decoding, hidden rows to the host
        _case("batcher_bf16_s16_r24_p100-600", "batcher", 16, 100, 600, 60, requests=24),
    ]


def _cost(c):
    """Rough milliseconds of a pass, to keep drawn cases no dearer than the largest listed one."""
    if c["model"] == "tiny":
        return 0.1 * (c["steps"] + 1)
    mean = (c["prefix_lo"] + c["prefix_hi"]) / 2
    n = max(c["streams"], c["requests"])
    rounds = -(-n // c["streams"])
    return 1 + n * mean * 0.0025 + rounds * c["steps"] * (0.48 + c["streams"] * (0.006 + (mean + c["steps"] / 2) * 2.2e-5))


def draw(rng):
    """One more session of the same ranges."""
    log_int = lambda lo, hi: int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))  # noqa: E731
    bound = 350.0
    while True:
        call = rng.choice(["decode_steps"] * 8 + ["decode_step", "decode_step_host", "prefill", "prefill", "prefill_tokens", "batcher"])
        model = "tiny" if rng.random() < 0.08 else "full"
        streams = log_int(1, 24 if call == "batcher" else 128)
        lo = log_int(N_COND + 6, 1900)
        hi = min(1900, int(lo * rng.uniform(1.0, 4.0)))
        steps = 0 if call.startswith("prefill") else log_int(16, 96)
        c = _case(None, call, streams, lo, hi, steps, model=model, weights=rng.choice(["bf16", "w8a16", "w4a16"]),
                  kv=rng.choice(["bf16", "bf16", "e4m3"]), top_k=rng.choice([0, 0, 30]) if call != "batcher" else 0,
                  logits=streams <= 16 and call != "batcher", requests=streams + rng.randint(1, streams) if call == "batcher" else 0)
        if hi + steps <= MAX_CONTEXT - 64 and _cost(c) <= bound:
            return c


# -- shapes ------------------------------------------------------------------------------------------
def _spread(n, lo, hi, shift=0.0):
    """n lengths spread evenly over lo..hi in a mixed order (golden-ratio sequence)."""
    if n == 1:
        return [(lo + hi) // 2]
    return [lo + int(((i * 0.6180339887498949 + shift) % 1.0) * (hi - lo + 1)) for i in range(n)]


def _lengths(case):
    """Prefix length and decode steps of every utterance of the session."""
    n = case["requests"] or case["streams"]
    p = _spread(n, case["prefix_lo"], case["prefix_hi"])
    if case["requests"]:        # requests ask for different amounts of audio
        return p, _spread(n, case["steps"] // 2, case["steps"] + case["steps"] // 2, 0.3)
    return p, [case["steps"]] * n


def _config(case):
    p, n = _lengths(case)
    pages = sorted(((a + b + 63) // 64 for a, b in zip(p, n)), reverse=True)
    kw = dict(wfmt=WEIGHTS[case["weights"]], kv_fmt=KV[case["kv"]], max_streams=case["streams"], max_context=MAX_CONTEXT,
              n_pages=sum(pages[:case["streams"]]))
    make = C.tiny_config if case["model"] == "tiny" else C.full_config
    cfg = make(**kw)
    text = TEXT_ROWS if case["call"] == "prefill_tokens" else 0
    return make(**kw, emb_rows=cfg.vocab + text if text else 0, max_pos=MAX_CONTEXT)


# -- weights -----------------------------------------------------------------------------------------
def _bits(x):
    return x.to(torch.bfloat16).view(torch.int16)


def _quantize(w, wfmt):
    """bf16 matrix -> (codes, scales) in the boundary formats."""
    if wfmt == C.W_BF16:
        return w.view(torch.int16), None
    f = w.float()
    if wfmt == C.W_INT8_PC:
        s = (f.abs().amax(1) / 127).to(torch.bfloat16)
        q = torch.clamp(torch.round(f / s.float()[:, None]), -127, 127).to(torch.int8)
        return q, s.view(torch.int16)
    n, k = f.shape
    g = f.view(n, k // 128, 128)
    s = (g.abs().amax(2) / 7).to(torch.bfloat16)
    u = (torch.clamp(torch.round(g / s.float()[:, :, None]), -8, 7) + 8).to(torch.int32).view(n, k // 8, 8)
    word = u[:, :, 0].clone()
    for j in range(1, 8):
        word |= u[:, :, j] << (4 * j)
    return word, s.view(torch.int16)


def _weights(cfg, gen):
    d, f, v = cfg.d_model, cfg.d_ff, cfg.vocab
    draw_ = lambda *shape, std=0.02, mean=0.0: (torch.randn(shape, generator=gen, device=DEV) * std + mean).to(torch.bfloat16)  # noqa: E731
    emb = draw_(cfg.n_emb_rows, d, std=1.0)
    if cfg.n_emb_rows > v:      # text ids share embeddings with semantic codes, so that they have successors too
        emb[v:] = emb[torch.randperm(v, generator=gen, device=DEV)[:cfg.n_emb_rows - v]]
    succ = torch.randperm(v, generator=gen, device=DEV)
    head = draw_(v, d).float()
    head[succ] += 0.8 * torch.nn.functional.normalize(emb[:v].float(), dim=1)
    w = {"tok_emb": _bits(emb), "pos_emb": _bits(draw_(cfg.max_pos, d)), "lnf_g": _bits(draw_(d, std=0.01, mean=1.0)),
         "lnf_b": _bits(draw_(d, std=0.01)), "head_w": _bits(head), "head_b": None}
    shapes = C.linear_shapes(cfg)
    per_layer = ["ln1_g", "ln1_b", "ln2_g", "ln2_b"] + [x + s for x in C.LINEARS for s in ("_w", "_s", "_b")]
    w.update({k: [] for k in per_layer})
    for _ in range(cfg.n_layer):
        for ln in ("ln1", "ln2"):
            w[ln + "_g"].append(_bits(draw_(d, std=0.01, mean=1.0)))
            w[ln + "_b"].append(_bits(draw_(d, std=0.01)))
        for lin in C.LINEARS:
            q, s = _quantize(draw_(*shapes[lin]), cfg.wfmt)
            w[lin + "_w"].append(q)
            w[lin + "_s"].append(s)
            w[lin + "_b"].append(_bits(draw_(shapes[lin][0])))
    return w, emb


# -- a session ---------------------------------------------------------------------------------------
_stream = None


def _engine_stream():
    """The engines of a process queue on one stream."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream(DEV)
    return _stream


def prepare(case, seed):
    cfg = _config(case)
    gen = torch.Generator(DEV).manual_seed(int(seed))
    weights, emb = _weights(cfg, gen)
    eng = B.TtsGpt(cfg, weights, DEV, stream=_engine_stream())
    p, n_dec = _lengths(case)
    s = {"case": case, "eng": eng, "n_dec": n_dec, "rows": case["streams"]}
    rows, steps, d, v = case["streams"], case["steps"], cfg.d_model, cfg.vocab
    if case["call"] == "prefill_tokens":
        s["cond"] = [torch.randn((N_COND, d), generator=gen, device=DEV).to(torch.bfloat16) for _ in p]
        s["text"] = [torch.randint(0, TEXT_ROWS, (x - N_COND,), generator=gen, device=DEV, dtype=torch.int32) for x in p]
    else:
        s["prefix"] = []
        for x in p:             # embeddings, the last one that of a token (start of audio)
            e = torch.randn((x, d), generator=gen, device=DEV).to(torch.bfloat16)
            e[-1] = emb[torch.randint(0, v, (1,), generator=gen, device=DEV)[0]]
            s["prefix"].append(e)
    if case["call"] != "batcher":
        on_host = case["call"] == "decode_step_host"
        s["uniforms"] = torch.rand((steps + 1, rows), generator=gen, device=DEV) if case["top_k"] > 1 else None
        s["first"] = {"tokens": torch.zeros(rows, dtype=torch.int32, device=DEV),
                      "logits": torch.zeros((rows, v), device=DEV) if case["logits"] else None,
                      "hidden": torch.zeros((rows, d), dtype=torch.bfloat16, device=DEV)}
        if steps:
            where = dict(pin_memory=True) if on_host else dict(device=DEV)
            s["out"] = {"tokens": torch.zeros((steps, rows), dtype=torch.int32, **where),
                        "logits": torch.zeros((steps, rows, v), **where) if case["logits"] else None,
                        "hidden": torch.zeros((steps, rows, d), dtype=torch.bfloat16, **where)}
            if on_host and s["uniforms"] is not None:
                s["uniforms_host"] = s["uniforms"].cpu().pin_memory()
    torch.cuda.synchronize()
    return s


def _batcher(s):
    """Submit every request, then take chunks of a quarter of a second until all are served."""
    case = s["case"]
    bt = ContinuousBatcher(s["eng"], keep_hidden=True)
    rid = [bt.submit(p, n) for p, n in zip(s["prefix"], s["n_dec"])]
    tokens, hidden = {r: [] for r in rid}, {r: [] for r in rid}
    while not bt.idle():
        for c in bt.run_chunk(12):
            tokens[c.rid].append(c.tokens)
            hidden[c.rid].append(c.hidden)
    tok = np.concatenate([x for r in rid for x in tokens[r]])
    hid = np.concatenate([x for r in rid for x in hidden[r]])
    return {"tokens": tok, "hidden": torch.from_numpy(hid.view(np.int16)).view(torch.bfloat16)}


def run(s):
    case, eng = s["case"], s["eng"]
    call, k, u, first = case["call"], case["top_k"], None, None
    if call == "batcher":
        return _batcher(s)
    u, first = s["uniforms"], s["first"]
    kw = dict(top_k=k, uniforms=None if u is None else u[0], out_tokens=first["tokens"], out_logits=first["logits"], out_hidden=first["hidden"])
    if call == "prefill_tokens":
        ids, _ = eng.prefill_tokens(s["cond"], s["text"], eng.cfg.vocab, 0, **kw)
    else:
        ids, _ = eng.prefill(s["prefix"], **kw)
    out = s.get("out")
    if call == "decode_steps":
        eng.decode_steps(ids, case["steps"], out["tokens"], top_k=k, uniforms=None if u is None else u[1:], out_logits=out["logits"],
                         out_hidden=out["hidden"])
    elif call in ("decode_step", "decode_step_host"):
        step = eng.decode_step if call == "decode_step" else eng.decode_step_host
        u = s.get("uniforms_host", u)
        lg = out["logits"]
        for i in range(case["steps"]):
            step(ids, out["tokens"][i], top_k=k, uniforms=None if u is None else u[i + 1], out_logits=None if lg is None else lg[i],
                 out_hidden=out["hidden"][i])
    for i in ids:
        eng.release_stream(i)
    return {"first": first, "steps": out}


# -- what a pass cannot do without --------------------------------------------------------------------
def work(case):
    cfg = _config(case)
    d, f, v, layers = cfg.d_model, cfg.d_ff, cfg.vocab, cfg.n_layer
    lin = 4 * d * d + 2 * d * f
    per = {"bf16": 2.0, "w8a16": 1.0, "w4a16": 0.5 + 2 / 128}[case["weights"]]
    weights = layers * (lin * per + (9 * d + f) * 2) + v * d * 2
    kv_tok = layers * (4 * d if case["kv"] == "bf16" else 2 * cfg.n_head * (64 + 4))
    row_flops = 2.0 * layers * lin
    out_row = d * 2 + 4 + (v * 4 if case["logits"] else 0)
    p, n = _lengths(case)
    b = weights + sum(x * (d * 2 + kv_tok) for x in p) + len(p) * out_row         # prefill: prefixes in, KV out
    fl = sum(x * row_flops + 2.0 * layers * d * x * (x + 1) + 2.0 * v * d for x in p)
    if case["requests"]:        # the first token of a request comes from its prefill
        n = [x - 1 for x in n]
    tot = sum(n)
    b += -(-tot // case["streams"]) * weights + sum(kv_tok * (x * k + k * (k + 1) // 2) for x, k in zip(p, n)) + tot * out_row
    fl += tot * (row_flops + 2.0 * v * d) + sum(4.0 * layers * d * (x * k + k * (k + 1) / 2) for x, k in zip(p, n))
    return {"bytes": float(b), "flops": float(fl)}


def tolerance(case):
    # two correct implementations round the bf16 operands of 24 layers along different histories: each is 0.5 % off
    # the exact logits; with 8-bit codes a value near a rounding edge takes the next code, one part in eight away.
    # A sampled token may differ where its uniform falls on an edge of the cumulative distribution.
    return {"rel": 2e-2 if case["kv"] == "e4m3" else 1e-2, "differ": 0.01 if case["top_k"] > 1 else 0.0}
