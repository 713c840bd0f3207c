"""What this library is measured on: calls and call sequences that a program with a QAQ cache issues.

A case is a dict of plain values with a "kind":

  decode      one generation step's attention over a filled cache: one query per (b,h), with or without the score
              row that feeds the attention window, or several queries at once ("queries" > 1: speculative or batched
              verification).  "widths" 0 = widths from the rules, otherwise one width for every token.
  prefill     a prompt has just been run: score window of its last queries, outlier thresholds, fused selection +
              quantization + packing, and the first decode step on the new cache.
  generate    a short session: the prompt's keys and values are quantized, then "steps" tokens are generated with the
              step captured in a CUDA graph (every layer's append + decode, the token count in device memory).
  adapt       the per-step loop of Section 4.2 of the paper launched from the host: append, decode with the score row,
              window update, lowering of widths over the whole cache; compaction at the end.
  requantize  a cache taken to lower widths and back up from the unquantized copy, compacted and read once.

Sizes are those of the configurations in paper_2403_04643_b200/synth.py (LLaMA-2-like head geometry) and of ragged
prompts around them.  The host-buffer entry points are left out: they are bound by the bus.
"""
from __future__ import annotations

import math

import torch

from paper_2403_04643_b200 import calibrate, qaq, synth

DEFAULTS = {"head_dim": 128, "batch": 1, "heads": 32, "window": 32, "alpha": 0.01, "dist": "normal"}


def _case(name, kind, **kw):
    c = dict(DEFAULTS, kind=kind, **kw)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: a short conversation on a small model, four heads of 64 channels
        _case("decode_small", "decode", heads=4, head_dim=64, tokens=500, window=5, queries=1, scores=True, widths=0),
        # one 7B-shaped layer, one request, the score row written for the window: the ordinary generation step
        _case("decode_7b", "decode", tokens=4096, queries=1, scores=True, widths=0),
        # the same layer in a serving batch of eight
        _case("decode_7b_batch8", "decode", batch=8, tokens=4096, queries=1, scores=False, widths=0),
        # a 13B-shaped layer with heavy tails: 5 % of the entries in the outlier lists
        _case("decode_13b_heavy", "decode", batch=4, heads=40, tokens=8192, window=64, alpha=0.05, dist="student3", queries=1,
              scores=False, widths=0),
        # one long-context request
        _case("decode_long", "decode", tokens=131072, queries=1, scores=True, widths=0),
        # four draft tokens verified in one call on the uniform 4-bit comparison cache
        _case("verify4_7b_batch8", "decode", batch=8, tokens=4096, queries=4, scores=False, widths=4),
        # a short ragged prompt, keys and values as the projection leaves them (token-major)
        _case("prefill_short", "prefill", tokens=333, layout="bthd"),
        # full 7B-shaped context, batch of eight
        _case("prefill_7b_batch8", "prefill", batch=8, tokens=4096, layout="bhtd"),
        # 13B-shaped, heavy tails, window of 64 queries, sequence beyond 4096 tokens
        _case("prefill_13b_heavy", "prefill", batch=4, heads=40, tokens=8192, window=64, alpha=0.05, dist="student3", layout="bhtd"),
        # a request of 1000 prompt tokens and 64 generated ones on four layers
        _case("generate_7b", "generate", tokens=1000, steps=64, layers=4),
        # the loop of Section 4.2 on one layer with four requests
        _case("adapt_7b_batch4", "adapt", batch=4, tokens=2048, steps=24),
        # memory pressure and release: widths down, up again, gaps closed
        _case("requantize_7b_batch4", "requantize", batch=4, tokens=4096),
    ]


def draw(rng):
    kind = rng.choice(["decode", "decode", "decode", "prefill", "prefill", "generate", "adapt", "requantize"])
    c = {"head_dim": rng.choice([128, 128, 128, 64, 32]), "heads": rng.choice([4, 8, 12, 32, 32, 40]), "batch": int(round(2 ** rng.uniform(0, 3)))}
    heavy = rng.random() < 0.25
    c["alpha"], c["dist"] = (0.05, "student3") if heavy else (rng.choice([0.01, 0.01, 0.02, 0.004]), "normal")
    c["window"] = rng.choice([1, 5, 16, 32, 32, 64])

    def tokens(lo, hi, most):
        """Token count spread over the logarithm of [lo, hi], odd ones among them, at most `most` entries per tensor."""
        hi = max(lo, min(hi, most // (c["batch"] * c["heads"] * c["head_dim"])))
        t = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return t if rng.random() < 0.7 else max(lo, t // 64 * 64)

    if kind == "decode":
        q = rng.choice([1, 1, 1, 2, 3, 4, 5, 8])
        most = 1 * 32 * 131072 * 128 if q == 1 else 8 * 32 * 4096 * 128 // (1 if q <= 4 else 2)
        return _case("", "decode", **c, tokens=tokens(64, 131072, most), queries=q, scores=q == 1 and rng.random() < 0.5,
                     widths=rng.choice([0, 0, 0, 2, 3, 4, 8]))
    if kind == "prefill":
        return _case("", "prefill", **c, tokens=tokens(40, 32768, 4 * 40 * 8192 * 128 // 2), layout=rng.choice(["bhtd", "bthd"]))
    if kind == "generate":
        return _case("", "generate", **c, tokens=tokens(40, 4096, 32 * 1024 * 128), steps=rng.choice([5, 17, 40, 64]), layers=rng.choice([1, 2, 4]))
    if kind == "adapt":
        return _case("", "adapt", **c, tokens=tokens(100, 4096, 4 * 32 * 2048 * 128), steps=rng.choice([4, 9, 24]))
    return _case("", "requantize", **c, tokens=tokens(64, 16384, 4 * 32 * 4096 * 128))


# ------------------------------------------------------------------------------------------------- inputs
def _workload(c, seed, tokens):
    heavy = c["dist"] == "student3"
    return synth.Workload("measured", c["batch"], c["heads"], c["head_dim"], tokens, c["window"], c["alpha"], dist=c["dist"],
                          outlier_frac=c["alpha"] if heavy else 0.01, seed=int(seed) * 1009 + 7)


def _hyper(c, tokens, attention_rows=False, low=False):
    """The calibrated hyper-parameters of the configuration the case belongs to, carried over to another length so
    that the mean widths stay about (4, 3) bits, or (2.2, 2.2) if low: scores fall like 1/T, and the budgets of the
    rules with them.  Attention rows of the window kernel are peakier than the synthetic ones, the budget looser."""
    name = "C4" if c["dist"] == "student3" else ("C3_low" if low else "C3")
    sS, sX, qn = calibrate.frozen(name)
    r = synth.CONFIGS[name[:2]].tokens / tokens
    f = (4.0 if low and name == "C4" else 1.0)
    return sS * r * f, sX * math.sqrt(r) * f * (ROWS_SPREAD if attention_rows else 1.0), qn


ROWS_SPREAD = 5.0


def _config(c, max_tokens):
    return qaq.make_config(c["batch"], c["heads"], c["head_dim"], max_tokens, 2, 8, c["window"], c["alpha"])


def _inputs(c, seed, tokens):
    """K, V, a query, and the attention window of the last tokens, on the GPU."""
    wl = _workload(c, seed, tokens)
    K, V = synth.make_kv(wl, device="cuda")
    ring, nvalid = synth.make_score_ring(wl, device="cuda")
    return wl, K, V, synth.make_query(wl, device="cuda"), ring, nvalid


def prepare(case, seed):
    return globals()["_prepare_" + case["kind"]](case, seed)


def run(state):
    return globals()["_run_" + state["case"]["kind"]](state)


# ------------------------------------------------------------------------------------------------- decode
def _prepare_decode(c, seed):
    T, BH, D = c["tokens"], c["batch"] * c["heads"], c["head_dim"]
    wl, K, V, q, ring, nvalid = _inputs(c, seed, T)
    cfg = _config(c, T)
    cache = qaq.Cache(cfg)
    thr = qaq.qaq_outlier_thresholds(cfg, K, V)
    if c["widths"]:
        bits = torch.full((BH, T), c["widths"], dtype=torch.uint8, device="cuda")
        qaq.qaq_quantize_append(cache, K, V, thr, bitsK=bits, bitsV=bits)
    else:
        pol = qaq.qaq_policy_from_hyper(*_hyper(c, T), T)
        qaq.qaq_quantize_append(cache, K, V, thr, policy=pol, ring=ring, nvalid=nvalid)
    n = c["queries"]
    if n > 1:
        q = torch.stack([synth.make_query(wl, step=i, device="cuda").view(BH, D) for i in range(n)], dim=1).contiguous()
    out = torch.empty((BH, n, D) if n > 1 else (BH, D), dtype=torch.float32, device="cuda")
    scores = torch.empty((BH, T), dtype=torch.float32, device="cuda") if c["scores"] else None
    return {"case": c, "cache": cache, "q": q, "out": out, "scores": scores, "scale": 1.0 / math.sqrt(D)}


def _run_decode(s):
    if s["case"]["queries"] > 1:
        return qaq.qaq_decode_attention_multi(s["cache"], s["q"], s["scale"], out=s["out"])
    out = qaq.qaq_decode_attention(s["cache"], s["q"], s["scale"], out=s["out"], scores_out=s["scores"])
    return out if s["scores"] is None else (out, s["scores"])


# ------------------------------------------------------------------------------------------------- prefill
def _prepare_prefill(c, seed):
    T, BH, D = c["tokens"], c["batch"] * c["heads"], c["head_dim"]
    wl = _workload(c, seed, T)
    K, V = synth.make_kv(wl, device="cuda")
    if c["layout"] == "bthd":
        K, V = (x.transpose(1, 2).contiguous().transpose(1, 2) for x in (K, V))
    Q = torch.stack([synth.make_query(wl, step=i, device="cuda").view(BH, D) for i in range(c["window"])], dim=1).contiguous()
    cfg = _config(c, T + 256)
    return {"case": c, "cfg": cfg, "cache": qaq.Cache(cfg), "K": K, "V": V, "Q": Q, "q": Q[:, -1].contiguous(),
            "policy": qaq.qaq_policy_from_hyper(*_hyper(c, T, attention_rows=True), T), "scale": 1.0 / math.sqrt(D),
            "thr": torch.empty((BH, 4), dtype=torch.float32, device="cuda"),
            "out": torch.empty((BH, D), dtype=torch.float32, device="cuda"),
            "scores": torch.empty((BH, T), dtype=torch.float32, device="cuda")}


def _run_prefill(s):
    cache, K, V = s["cache"], s["K"], s["V"]
    cache.reset()
    ring, nvalid = qaq.qaq_prefill_window(s["cfg"], s["Q"], K, s["scale"])
    thr = qaq.qaq_outlier_thresholds(s["cfg"], K, V, s["thr"])
    qaq.qaq_quantize_append(cache, K, V, thr, policy=s["policy"], ring=ring, nvalid=nvalid)
    out = qaq.qaq_decode_attention(cache, s["q"], s["scale"], out=s["out"], scores_out=s["scores"])
    return thr, ring, nvalid, out, s["scores"]


# ------------------------------------------------------------------------------------------------- generate
def _prepare_generate(c, seed):
    T, n, B, H, D, W = c["tokens"], c["steps"], c["batch"], c["heads"], c["head_dim"], c["window"]
    cfg = _config(c, T + n + 1)
    scale = 1.0 / math.sqrt(D)
    policy = qaq.qaq_policy_from_hyper(*_hyper(c, T), T)
    step_in = torch.zeros((c["layers"], 3, B, H, D), dtype=torch.float16, device="cuda")     # k, v, q of one step
    step_out = torch.zeros((c["layers"], B * H, D), dtype=torch.float32, device="cuda")
    no_score = torch.zeros((B, H, W, 1), dtype=torch.float32, device="cuda")
    no_rows = torch.zeros((B, H, 1), dtype=torch.uint8, device="cuda")
    layers, new = [], []
    for l in range(c["layers"]):
        wl, K, V, _, ring, nvalid = _inputs(c, seed * 64 + l, T)
        k1, v1 = synth.make_kv(synth.scaled(wl, seed=wl.seed + 500_000_000), device="cuda", tokens=n)
        q1 = torch.stack([synth.make_query(wl, step=i, device="cuda") for i in range(n)])
        new.append(torch.stack([k1.permute(2, 0, 1, 3), v1.permute(2, 0, 1, 3), q1], dim=1))
        layers.append({"cache": qaq.Cache(cfg), "K": K, "V": V, "ring": ring, "nvalid": nvalid,
                       "thr": torch.empty((B * H, 4), dtype=torch.float32, device="cuda")})
    # (the captured step reads no_score and no_rows at every replay: the program keeps them as long as the graph)
    s = {"case": c, "cfg": cfg, "layers": layers, "policy": policy, "step_in": step_in, "step_out": step_out, "no_score": no_score, "no_rows": no_rows,
         "new": torch.stack(new, dim=1).contiguous(), "outs": torch.zeros((n, c["layers"], B * H, D), dtype=torch.float32, device="cuda")}

    def step():
        for l, L in enumerate(layers):
            k, v, q = step_in[l]
            qaq.qaq_stream_append(L["cache"], k, v, L["thr"], policy=policy, score_col=no_score, nvalid=no_rows)
            qaq.qaq_stream_decode(L["cache"], q, scale, step_out[l])

    _quantize_prompts(s)
    step()                                     # once on the stream, then captured
    torch.cuda.synchronize()
    s["graph"] = torch.cuda.CUDAGraph()
    with torch.cuda.graph(s["graph"]):
        step()
    for L in layers:
        qaq.qaq_stream_end(L["cache"])
    return s


def _quantize_prompts(s):
    for L in s["layers"]:
        L["cache"].reset()
        qaq.qaq_outlier_thresholds(s["cfg"], L["K"], L["V"], L["thr"])
        qaq.qaq_quantize_append(L["cache"], L["K"], L["V"], L["thr"], policy=s["policy"], ring=L["ring"], nvalid=L["nvalid"])
        qaq.qaq_stream_begin(L["cache"])


def _run_generate(s):
    _quantize_prompts(s)
    for i in range(s["case"]["steps"]):
        s["step_in"].copy_(s["new"][i])
        s["graph"].replay()
        s["outs"][i].copy_(s["step_out"])
    for L in s["layers"]:
        qaq.qaq_stream_end(L["cache"])
    return s["outs"]


# ------------------------------------------------------------------------------------------------- adapt
def _prepare_adapt(c, seed):
    T, n, B, H, D, W = c["tokens"], c["steps"], c["batch"], c["heads"], c["head_dim"], c["window"]
    wl, K, V, _, ring0, nvalid0 = _inputs(c, seed, T + n)
    ring0, nvalid0 = ring0[..., :T].contiguous(), nvalid0[..., :T].contiguous()
    cfg = _config(c, 2 * (T + n))              # room for tiles that move when their widths change
    return {"case": c, "cfg": cfg, "cache": qaq.Cache(cfg), "K": K, "V": V, "ring0": ring0, "nvalid0": nvalid0, "hyper": _hyper(c, T),
            "q": torch.stack([synth.make_query(wl, step=i, device="cuda") for i in range(n)]), "scale": 1.0 / math.sqrt(D),
            "thr": torch.empty((B * H, 4), dtype=torch.float32, device="cuda"),
            "ring": torch.zeros((B, H, W, T + n), dtype=torch.float32, device="cuda"),
            "nvalid": torch.zeros((B, H, T + n), dtype=torch.uint8, device="cuda"),
            "new_ring": torch.zeros((B, H, W, 1), dtype=torch.float32, device="cuda"),
            "new_nvalid": torch.zeros((B, H, 1), dtype=torch.uint8, device="cuda"),
            "scores": torch.empty((B * H * (T + n),), dtype=torch.float32, device="cuda"),
            "outs": torch.zeros((n, B * H, D), dtype=torch.float32, device="cuda")}


def _run_adapt(s):
    c, cache, K, V, ring, nvalid, thr = s["case"], s["cache"], s["K"], s["V"], s["ring"], s["nvalid"], s["thr"]
    T0, n, B, H, W = c["tokens"], c["steps"], c["batch"], c["heads"], c["window"]
    cache.reset()
    ring.zero_()
    nvalid.zero_()
    ring[..., :T0] = s["ring0"]
    nvalid[..., :T0] = s["nvalid0"]
    qaq.qaq_outlier_thresholds(s["cfg"], K[:, :, :T0], V[:, :, :T0], thr)
    qaq.qaq_quantize_append(cache, K[:, :, :T0], V[:, :, :T0], thr, policy=qaq.qaq_policy_from_hyper(*s["hyper"], T0),
                            ring=s["ring0"], nvalid=s["nvalid0"])
    for i in range(n):
        t = T0 + i
        policy = qaq.qaq_policy_from_hyper(*s["hyper"], t + 1)
        qaq.qaq_quantize_append(cache, K[:, :, t:t + 1], V[:, :, t:t + 1], thr, policy=policy, ring=s["new_ring"], nvalid=s["new_nvalid"])
        row = s["scores"][:B * H * (t + 1)].view(B * H, t + 1)
        qaq.qaq_decode_attention(cache, s["q"][i], s["scale"], out=s["outs"][i], scores_out=row)
        ring[:, :, t % W, :t + 1] = row.view(B, H, t + 1)
        nvalid[:, :, :t + 1] += 1
        nvalid.clamp_(max=W)
        qaq.qaq_requantize_down(cache, policy=policy, ring=ring, nvalid=nvalid)
    qaq.qaq_cache_compact(cache)
    return s["outs"], ring, nvalid


# ------------------------------------------------------------------------------------------------- requantize
def _prepare_requantize(c, seed):
    T, BH, D = c["tokens"], c["batch"] * c["heads"], c["head_dim"]
    _, K, V, q, ring, nvalid = _inputs(c, seed, T)
    cfg = _config(c, 2 * T + 64)               # room for the tiles that grow again
    cache = qaq.Cache(cfg)
    thr = qaq.qaq_outlier_thresholds(cfg, K, V)
    high, low = (qaq.qaq_policy_from_hyper(*_hyper(c, T, low=x), T) for x in (False, True))
    qaq.qaq_quantize_append(cache, K, V, thr, policy=high, ring=ring, nvalid=nvalid)
    return {"case": c, "cache": cache, "K": K, "V": V, "q": q, "ring": ring, "nvalid": nvalid, "thr": thr, "high": high, "low": low,
            "scale": 1.0 / math.sqrt(D), "out": torch.empty((2, BH, D), dtype=torch.float32, device="cuda"),
            "scores": torch.empty((2, BH, T), dtype=torch.float32, device="cuda")}


def _run_requantize(s):
    cache = s["cache"]
    qaq.qaq_requantize_down(cache, policy=s["low"], ring=s["ring"], nvalid=s["nvalid"])
    qaq.qaq_decode_attention(cache, s["q"], s["scale"], out=s["out"][0], scores_out=s["scores"][0])
    qaq.qaq_requantize(cache, s["K"], s["V"], s["thr"], policy=s["high"], ring=s["ring"], nvalid=s["nvalid"])
    qaq.qaq_cache_compact(cache)
    qaq.qaq_decode_attention(cache, s["q"], s["scale"], out=s["out"][1], scores_out=s["scores"][1])
    return s["out"], s["scores"]


# ------------------------------------------------------------------------------------------------- work, tolerance
def work(c):
    """Bytes each pass cannot do without (inputs read once, results written once; packed codes at the nominal mean
    widths) and the multiply-adds of its contractions."""
    T, BH, D, W = c["tokens"], c["batch"] * c["heads"], c["head_dim"], c["window"]

    def packed(th, bits):                       # codes, width + min + max per token and tensor, outlier entries
        return th * (D * sum(bits) / 8 + 10 + 2 * D * c["alpha"] * 4)

    io = BH * D * (2 + 4)                       # a query in, a result out
    mean = (4, 3)
    if c["kind"] == "decode":
        bits = (c["widths"],) * 2 if c["widths"] else mean
        n = c["queries"]
        return {"bytes": packed(BH * T, bits) + n * io + (4 * BH * T if c["scores"] else 0), "flops": 4.0 * n * BH * T * D}
    if c["kind"] == "prefill":
        return {"bytes": BH * T * (4 * D + 4 * W + 1 + 4) + 2 * packed(BH * T, mean) + io + BH * W * D * 2,
                "flops": BH * T * D * (2.0 * W + 4.0)}
    if c["kind"] == "generate":
        n = c["steps"]
        tokens = sum(T + i + 1 for i in range(n))
        prompt = BH * T * (4 * D + 4 * W + 1) + packed(BH * T, mean)
        step = packed(BH * tokens, mean) + n * (packed(BH, (4, 8)) + 4 * BH * D + io)
        return {"bytes": c["layers"] * (prompt + step), "flops": 4.0 * c["layers"] * BH * tokens * D}
    if c["kind"] == "adapt":
        n = c["steps"]
        tokens = sum(T + i + 1 for i in range(n))
        prompt = BH * T * (4 * D + 4 * W + 1) + packed(BH * T, mean)
        # per step: the packed cache and every window row read, the score row written once as such and once into the
        # window, ranges and widths read and the rows-per-token counts updated
        step = packed(BH * tokens, mean) + BH * tokens * (4 * W + 8 + 10 + 2) + n * (packed(BH, (4, 8)) + 4 * BH * D + io)
        return {"bytes": prompt + step, "flops": 4.0 * BH * tokens * D}
    low = (2.2, 2.2)
    ranges = 2 * BH * T * (4 * W + 1 + 10 + 2)
    codes = lambda b: BH * T * D * sum(b) / 8  # noqa: E731
    # down: old codes read, new written; up: unquantized rows read, new codes written; two reads of the cache
    return {"bytes": ranges + codes(mean) + codes(low) + 4 * BH * T * D + codes(mean) + packed(BH * T, low) + packed(BH * T, mean) +
            2 * (io + 4 * BH * T), "flops": 8.0 * BH * T * D}


def tolerance(c):
    # Measured against attention in binary64 on the reconstructed keys and values, about four times of it stated: one
    # query 1e-5 to 5.3e-5 of the norm, single entries up to 1.6e-3 of the root mean square; several queries, whose value
    # weights share one fixed-point scale, up to 1.4e-4 and 3.6e-3.
    if c["kind"] == "decode":
        return {"rel": 2.5e-4, "max": 6.5e-3} if c["queries"] == 1 else {"rel": 6e-4, "max": 1.5e-2}
    # Where widths follow from scores that were computed before, a score that comes out one unit in the last place
    # higher can give a token one bit more: its share of one result then moves by a fraction of a quantization step.
    return {"rel": 5e-4, "max": 2e-2}
