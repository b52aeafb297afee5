"""Performance cases of the VATP library: the passes a serving program makes through its public calls.

A case is one pass of one of these kinds ("path"):

  prefill  what happens to one layer when a prompt has arrived: a scoring call, vatp_select, and the compaction that fits
           the indicator (vatp_compact, or vatp_compact_window with a history window)
  score    the scoring call alone.  For the long or wide prompts: among 10^5 or more scores one is likely to lie within
           rounding of its unit's budget boundary, and the kept set is then not the same for every correct program
  prune    selection and compaction of scores that are already there: integer work and copies, exact
  decode   `steps` generation steps over `layers` layer caches, visited in turn

"call" names the scoring call: "scores" (vatp_prefill_scores), "attention" (vatp_prefill_attention_scores: the layer's
attention output too) or "lse" (vatp_prefill_scores_from_lse: the caller's attention forward left its row normalisers).
"""
from __future__ import annotations

import math

import torch

from paper_2406_12335_b200 import synth, vatp as V


def listed():
    return [
        # the smallest job there is: one short fp32 prompt, two heads (launch and latency bound)
        _prefill("prefill_tiny_f32", "scores", "f32", 1, 2, 64, 512, 256, n_recent=32),
        # the benchmark's layer: LLaMA2-7B shape, 4K prompt, half of it kept
        _score("score_4k", "scores", "bf16", 1, 32, 128, 4096, 2048, n_recent=128),
        # heads of 64 channels, a prompt of odd length, Appendix A's H2O split of a 50 % budget
        _prefill("prefill_d64", "scores", "bf16", 1, 16, 64, 1531, 766, n_sink=20, n_recent=383),
        # history window (Eq. 3): one prompt of the 2K windowed workload
        _prefill("prefill_window", "scores", "bf16", 1, 32, 128, 2048, 1024, n_recent=10, window=256),
        # grouped queries, 32 query / 8 KV heads, attention output wanted too; odd prompt length
        _prefill("prefill_gqa_attention", "attention", "bf16", 2, 32, 128, 3001, 1500, kv_heads=8, n_recent=128),
        # a wide batch of 8K prompts, as one layer of the 32-layer stack
        _score("score_8k_b8", "scores", "bf16", 8, 32, 128, 8192, 1638, n_recent=256),
        # the longest prompt, attention forward and scores in one call
        _score("attention_32k", "attention", "bf16", 1, 32, 128, 32768, 3277, n_recent=512),
        # selection and compaction of the wide batch
        _case("prune_8k_b8", "prune", "bf16", 8, 32, 128, 8192, 1638, n_recent=256),
        # generation at the benchmark's shape: eight layers in turn, every step after the one before (the next layer's
        # query comes out of this one), replayed from a graph
        _decode("decode_2k", "bf16", 1, 32, 128, 2048, 8, 4, graph=True, n_recent=128),
        # a wide batch stepped over independent caches, launches allowed to run side by side
        _decode("decode_1638_b8", "bf16", 8, 32, 128, 1638, 4, 2, graph=True, overlap=True, n_recent=256),
        # the windowed workload's steps: probabilities leave the window as they enter it
        _decode("decode_window", "bf16", 16, 32, 128, 1024, 2, 4, graph=True, n_recent=10, window=256),
        # one grouped-query sequence, calls issued one by one from the program without a graph
        _decode("decode_gqa_eager", "bf16", 1, 32, 128, 2048, 8, 2, kv_heads=8, n_recent=128),
    ]


def draw(rng):
    """Another case of the same ranges.  The caps keep every one cheaper than the longest listed prompt."""
    path = rng.choice(("prefill", "prefill", "score", "score", "prune", "decode", "decode", "decode"))
    dtype, d = rng.choice((("bf16", 128),) * 6 + (("bf16", 64),) * 2 + (("f32", 64), ("f32", 128)))
    main = (dtype, d) == ("bf16", 128)                  # the other combinations serve smaller models
    kv = rng.choice((0, 0, 8)) if main else 0
    heads = 32 if kv else rng.choice((2, 8, 12, 16, 32))
    window = rng.choice((0, 0, 0, 256, 400))
    if path == "decode":
        budget = _log(rng, 128, 4096)
        batch = max(1, min(_log(rng, 1, 16), (1 << 20 if main else 1 << 18) // (heads * budget)))
        layers = 2 if window else rng.choice((2, 4, 8))
        return _decode("", dtype, batch, heads, d, budget, layers, rng.choice((1, 2, 4)), kv_heads=kv, window=window,
                       graph=rng.random() < 0.7, overlap=rng.random() < 0.4, n_recent=min(rng.choice((10, 32, 128)), budget // 2))
    most = 1 << 15 if path == "prefill" else 1 << 19 if main else 1 << 16     # cached rows over all heads
    T = _log(rng, 257, (4096 if path == "prefill" else 16384) if main else 2048)
    batch = max(1, min(_log(rng, 1, 12), most // ((kv or heads) * T)))
    heads = heads if kv else min(heads, most // T)
    budget = math.floor(rng.choice((0.1, 0.2, 0.25, 0.5, 0.5)) * T + 0.5)
    sinks = min(rng.choice((0, 0, 2, 20)), budget // 4)
    recent = min(rng.choice((10, 32, 128, budget // 2)), budget - sinks)
    call = rng.choice(("scores", "scores", "attention") if kv else ("scores", "scores", "lse", "attention") if dtype == "bf16" else ("scores", "lse"))
    if path == "prune":
        return _case("", path, dtype, batch, kv or heads, d, T, budget, window=window, n_sink=sinks, n_recent=recent)
    norm = rng.choice(("l1",) * 6 + ("l2", "linf"))
    return (_prefill if path == "prefill" else _score)("", call, dtype, batch, heads, d, T, budget, kv_heads=kv, window=window,
                                                       n_sink=sinks, n_recent=recent, norm=norm)


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _case(name, path, dtype, batch, heads, head_dim, seq_len, budget, *, kv_heads=0, window=0, n_sink=0, n_recent=0,
          norm="l1", **more):
    c = {"path": path, "dtype": dtype, "batch": batch, "heads": heads, "kv_heads": kv_heads, "head_dim": head_dim, "seq_len": seq_len,
         "budget": budget, "n_sink": n_sink, "n_recent": n_recent, "window": window, "norm": norm, **more}
    return {"name": name, **c} if name else c


def _prefill(name, call, *a, **kw):
    return _case(name, "prefill", *a, call=call, **kw)


def _score(name, call, *a, **kw):
    return _case(name, "score", *a, call=call, **kw)


def _decode(name, dtype, batch, heads, head_dim, budget, layers, steps, *, graph=False, overlap=False, **kw):
    # the caches stand for prompts twice as long as the budget
    return _case(name, "decode", dtype, batch, heads, head_dim, 2 * budget, budget, layers=layers, steps=steps, graph=graph,
                 overlap=overlap, **kw)


# ------------------------------------------------------------------------------------------------ inputs
def _workload(case, seed):
    """The synthetic workload of a case; the seed goes where the generators take the workload's number."""
    return synth.Workload(1000 + seed, "case", case["dtype"], case["batch"], case["kv_heads"] or case["heads"], 1, case["head_dim"],
                          case["seq_len"], case["budget"], case["n_sink"], case["n_recent"], "window" if case["window"] else "h2o",
                          case["window"], case.get("steps", 0))


def _params(case, **kw):
    return V.make_params(batch=case["batch"], heads=case["heads"], kv_heads=case["kv_heads"], seq_len=case["seq_len"],
                         head_dim=case["head_dim"], dtype=case["dtype"], budget=case["budget"], n_sink=case["n_sink"],
                         n_recent=case["n_recent"], indicator="window" if case["window"] else "h2o", window=case["window"], norm=case["norm"], **kw)


def _grouped(wl, case, q_shape, layer):
    """Queries for `heads` query heads that lean towards their KV head's sinks."""
    u = synth.sink_direction(wl, layer, "cuda").repeat_interleave(case["heads"] // case["kv_heads"], dim=1)
    g = torch.Generator(device="cuda").manual_seed(977 * wl.cid + 31 * layer + len(q_shape))
    q = torch.randn(q_shape, generator=g, device="cuda")
    lean = u if q_shape[-2] != case["heads"] else u.squeeze(2)
    return (q + synth.sink_alpha(wl) * lean).to(wl.torch_dtype)


def _qkv(wl, case, layer=0):
    q, k, v = synth.prefill_inputs(wl, layer, "cuda")
    if case["kv_heads"]:
        q = _grouped(wl, case, (case["batch"], case["heads"], case["seq_len"], case["head_dim"]), layer)
    return q, k, v


def _indicator(case, seed):
    """Indicators as a prompt leaves them: two sinks that take a quarter of the attention, the rest falling with the
    position (a late token has been seen by few queries), log-normal around that."""
    b, h, T = case["batch"], case["kv_heads"] or case["heads"], case["seq_len"]
    g = torch.Generator(device="cuda").manual_seed(31337 + seed)
    age = torch.arange(T, 0, -1, dtype=torch.float64, device="cuda")
    seen = (1.0 / age.flip(0)).flip(0).cumsum(0).flip(0).float()     # sum of 1/j over the queries from the key's own on
    acc = seen * torch.exp(0.3 * torch.randn(b, h, T, generator=g, device="cuda"))
    acc[:, :, :2] += T / 8
    return acc.contiguous()


def _row_normalisers(case, q, k):
    """Natural-log row normalisers of every causal row (rows before a history window are never read: zeros there)."""
    G = q.shape[1] // k.shape[1]
    T, w = case["seq_len"], case["window"]
    first = max(T - w, 0) if w else 0
    lse = torch.zeros(q.shape[:3], device="cuda")
    ahead = torch.arange(T, device="cuda")
    for b in range(q.shape[0]):
        for h in range(q.shape[1]):
            kt = k[b, h // G].float().t()
            for r in range(first, T, 4096):
                rows = slice(r, min(r + 4096, T))
                s = (q[b, h, rows].float() @ kt) * case["head_dim"] ** -0.5
                s.masked_fill_(ahead[None, :] > ahead[rows, None], -math.inf)
                lse[b, h, rows] = torch.logsumexp(s, dim=1)
    return lse


def prepare(case, seed):
    path, wl = case["path"], _workload(case, seed)
    st = {"path": path, "window": case["window"], "status": torch.zeros(1, dtype=torch.int32, device="cuda")}
    if path == "decode":
        return _prepare_decode(st, case, wl, seed)
    b, hq, h, T, B = case["batch"], case["heads"], case["kv_heads"] or case["heads"], case["seq_len"], case["budget"]
    st["p"] = p = _params(case)
    q, st["k"], st["v"] = _qkv(wl, case)
    f32 = dict(dtype=torch.float32, device="cuda")
    if path == "prune":
        st["attn_acc"] = _indicator(case, seed)
        st["vnorm"] = st["v"].float().abs().sum(-1)
        st["score"] = st["attn_acc"] * st["vnorm"]
        if case["window"]:
            st["q"], st["lse"] = q, _row_normalisers(case, q, st["k"])
    else:
        st["q"], st["call"] = q, case["call"]
        for name in ("attn_acc", "vnorm", "score"):
            st[name] = torch.empty(b, h, T, **f32)
        if case["call"] == "lse":
            st["lse"] = _row_normalisers(case, q, st["k"])
        elif case["window"]:
            st["lse"] = torch.zeros(b, hq, T, **f32)       # rows before the window are not written
        if case["call"] == "attention":
            st["attn_out"] = torch.empty_like(q)
        st["workspace"] = torch.empty(max(V.vatp_workspace_bytes(p), 256), dtype=torch.uint8, device="cuda")
    if path != "score":
        st["kept"] = torch.empty(b, h, B, dtype=torch.int32, device="cuda")
        st["cache"] = V.Cache(p)
    return st


def _prepare_decode(st, case, wl, seed):
    b, hq, h, B = case["batch"], case["heads"], case["kv_heads"] or case["heads"], case["budget"]
    T, d, steps = case["seq_len"], case["head_dim"], case["steps"]
    st["p"] = _params(case, decode_overlap=case["overlap"])
    st["steps"], st["layers"] = steps, []
    for layer in range(case["layers"]):
        q, k, v = _qkv(wl, case, layer)
        acc, vnorm = _indicator(case, seed * 64 + layer), v.float().abs().sum(-1)
        kept = torch.empty(b, h, B, dtype=torch.int32, device="cuda")
        cache = V.Cache(st["p"])
        V.vatp_select(st["p"], acc * vnorm, kept)
        if case["window"]:
            V.vatp_compact_window(st["p"], q, k, v, _row_normalisers(case, q, k), acc, vnorm, kept, cache)
        else:
            V.vatp_compact(st["p"], k, v, acc, vnorm, kept, cache)
        dq, dk, dv = synth.decode_inputs(wl, layer, steps, "cuda")
        if case["kv_heads"]:
            dq = _grouped(wl, case, (steps, b, hq, d), layer)
        out = torch.empty(steps, b, hq, d, dtype=wl.torch_dtype, device="cuda")
        evicted = torch.empty(steps, b, h, dtype=torch.int32, device="cuda")
        # one token's buffers are views that the program makes once
        st["layers"].append((cache, list(zip(dq, dk, dv, out, evicted)), out, evicted))
    torch.cuda.synchronize()
    if case["graph"]:
        st["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(st["graph"]):
            _steps(st)
    return st


# ------------------------------------------------------------------------------------------------ one pass
def _steps(st):
    for s in range(st["steps"]):
        for cache, tokens, _, _ in st["layers"]:
            q, k, v, out, evicted = tokens[s]
            V.vatp_decode_step(st["p"], cache, q, k, v, out, evicted_pos=evicted, dev_status=st["status"])


def _cache_out(cache):
    # (acc is the float image of the windowed state's integer sums)
    got = [cache.k_cache, cache.v_cache, cache.acc, cache.vnorm, cache.pos]
    return got if cache.ring is None else got + [cache.ring]


def run(st):
    if st["path"] == "decode":
        if "graph" in st:
            st["graph"].replay()
        else:
            _steps(st)
        return [st["status"]] + [[out, evicted] + _cache_out(cache) for cache, _, out, evicted in st["layers"]]
    p, q, k, v = st["p"], st.get("q"), st["k"], st["v"]
    acc, vnorm, score, lse = st["attn_acc"], st["vnorm"], st["score"], st.get("lse")
    got = {"status": st["status"]}
    if st["path"] != "prune":
        to = dict(attn_acc=acc, vnorm=vnorm, score=score, workspace=st["workspace"], dev_status=st["status"])
        if st["call"] == "lse":
            V.vatp_prefill_scores_from_lse(p, q, k, v, lse, **to)
        elif st["call"] == "attention":
            V.vatp_prefill_attention_scores(p, q, k, v, st["attn_out"], lse_out=lse, **to)
            got["attn_out"] = st["attn_out"]
        else:
            V.vatp_prefill_scores(p, q, k, v, lse_out=lse, **to)
        got.update(attn_acc=acc, vnorm=vnorm, score=score, lse=lse)
    if st["path"] != "score":
        V.vatp_select(p, score, st["kept"], dev_status=st["status"])
        if st["window"]:
            V.vatp_compact_window(p, q, k, v, lse, acc, vnorm, st["kept"], st["cache"], dev_status=st["status"])
        else:
            V.vatp_compact(p, k, v, acc, vnorm, st["kept"], st["cache"], dev_status=st["status"])
        got.update(kept=st["kept"], cache=_cache_out(st["cache"]))
    return got


# ------------------------------------------------------------------------------------------------ what a pass needs
def work(case):
    """Inputs read and outputs written once; each query-key product of the causal half (or of the history window's
    rows) once for the scores, and once more each for the attention output's two products."""
    b, hq, h, T, B = case["batch"], case["heads"], case["kv_heads"] or case["heads"], case["seq_len"], case["budget"]
    d, eb, w = case["head_dim"], 4 if case["dtype"] == "f32" else 2, min(case["window"], case["seq_len"])
    row, units, q_units = d * eb, b * h, b * hq
    if case["path"] == "decode":
        n = case["layers"] * case["steps"]
        # K, V; indicator in and out, norm, position; with a window the 64-bit sums and the ring row that leaves and enters
        per_slot = 2 * row + 16 + (20 if w else 0)
        return {"bytes": n * (units * (B + 1) * per_slot + 2 * q_units * row), "flops": n * q_units * (B + 1) * 4.0 * d}
    nbytes = flops = 0.0
    pairs = w * T - w * (w - 1) / 2 if w else T * (T + 1) / 2
    if case["path"] != "prune":
        q_rows = T if not w or case["call"] == "attention" else w
        nbytes += q_units * q_rows * row + units * (2 * T * row + 12 * T)
        flops += q_units * 2.0 * d * pairs
        if case["call"] == "attention":
            flops += q_units * 2.0 * d * T * (T + 1) / 2
            flops += q_units * 2.0 * d * (T * (T + 1) / 2 - pairs)
            nbytes += q_units * T * row
    if case["path"] != "score":
        kept = min(B, T)
        nbytes += units * (4 * T + 4 * B + 4 * kept * row + 12 * kept)
        if w:
            nbytes += units * (w * kept * 4 + 8 * kept) + q_units * (w * row + 4 * w)
            flops += q_units * 2.0 * d * w * kept
    return {"bytes": nbytes, "flops": flops}


def tolerance(case):
    bf16 = case["dtype"] == "bf16"
    if case["path"] == "prune" and not case["window"]:
        return "exact"
    if case["path"] == "decode" or case.get("call") == "attention":
        # output rows in bf16 (measured against 64 bits: 2.4e-3, largest 0.03); whole values: an eviction within rounding
        return {"rel": 1e-2, "max": 0.12, "differ": 1e-3} if bf16 else {"rel": 1e-5, "max": 1e-3, "differ": 1e-3}
    # sums of probabilities in 32 bits.  bf16: the exponential is good to 7.5e-5 (indicators measured against 64 bits:
    # 4.7e-5); fp32: 1e-7, largest 2e-7, more where a logit's own rounding shows in a single probability of the window
    return {"rel": 2e-4, "max": 4e-4} if bf16 else {"rel": 2e-6, "max": 2e-5}
