"""What this framework is used for, as cases that can be timed: decode steps over a
mixed-precision cache from the smallest to the largest batch and context, prompts
written into the cache, several queries of a sequence at once, a mode per head, routed
calls and the router's decisions alone.

A case's sizes are this repository's workloads (workloads.py: tiny, 160m, 1p3b,
gqa_long, sweep) and the layouts its tests use.  Decoding cases are captured in a CUDA
graph once, as a serving loop keeps them, and every pass continues from the end of the
same prompts: the cache's bookkeeping is put back to where the prompts ended (as for
another continuation of the same prompt), then the steps run.
"""
import math

import torch

from paper_2607_06601_gb300 import trr

BITS = (2, 4, 8, 16)
SKIP, LOCAL, FULL = 0, 1, 2

# Router mixes of the workloads: probabilities of the widths 2, 4, 8, 16 and of the modes
# skip, local, full; whether 1 % of the channels are outliers (x8); gaps (lo, hi) between
# tokens forced to 16 bits (sentence starts), or None.
MIXES = {
    "tiny": ((0.25, 0.25, 0.25, 0.25), (1 / 3, 1 / 3, 1 / 3), False, None),
    "160m": ((0.20, 0.40, 0.30, 0.10), (0.20, 0.50, 0.30), True, None),
    "1p3b": ((0.25, 0.45, 0.25, 0.05), (0.20, 0.55, 0.25), False, (10, 30)),
    "gqa_long": ((0.50, 0.45, 0.00, 0.05), (0.15, 0.70, 0.15), False, None),
}

# Head layouts: query heads, KV heads, head size, quantiser group.
SHAPES = {
    "mha12": (12, 12, 64, 32),      # 160m
    "mha32": (32, 32, 64, 32),      # 1p3b, sweep
    "gqa32": (32, 8, 128, 64),      # gqa_long
    "gqa4": (4, 2, 64, 32),         # tiny
    "mha8w": (8, 8, 128, 64),       # layouts of the tests
    "gqa8w": (8, 2, 128, 64),
    "gqa12": (12, 4, 64, 64),
}


def _case(name, kind, shape, mix, **kw):
    c = {"name": name, "kind": kind, "shape": shape, "mix": mix, "page": 32, "layers": 1, "batch": 1,
         "ctx_lo": 0, "ctx_hi": 0, "window": 256, "steps": 1, "chunk": 1}
    c.update(kw)
    return c


def listed():
    return [
        # the smallest work: two short sequences generated token by token from an empty
        # cache (a test or a demo of the framework); nothing but latency
        _case("generate_tiny", "generate", "gqa4", "tiny", page=16, batch=2, ctx_lo=37, ctx_hi=130, window=32),
        # one user of a 24-layer model: the decode step that latency is quoted for
        _case("decode_sweep_b1", "decode", "mha32", "160m", layers=24, batch=1, ctx_lo=4096, ctx_hi=4096, steps=4),
        # the benchmark's decode step: the 160M model, batch 32, contexts of 2048
        _case("decode_160m", "decode", "mha12", "160m", layers=12, batch=32, ctx_lo=2048, ctx_hi=2048, steps=4),
        # the 1.3B shape with ragged contexts, as a server's running batch has them
        _case("decode_1p3b", "decode", "mha32", "1p3b", layers=4, batch=64, ctx_lo=1024, ctx_hi=8192, window=512,
              steps=2),
        # long contexts with grouped queries
        _case("decode_gqa_long", "decode", "gqa32", "gqa_long", layers=3, batch=16, ctx_lo=32768, ctx_hi=32768,
              window=1024, steps=4),
        # the largest batch of the sweep: throughput serving
        _case("decode_sweep_b256", "decode", "mha32", "160m", layers=3, batch=256, ctx_lo=4096, ctx_hi=4096, steps=2),
        # prompts written into an empty cache, 1024 tokens a call: quantise-on-write
        _case("prefill_160m", "prefill", "mha12", "160m", layers=4, batch=8, ctx_lo=2000, ctx_hi=2048),
        # one long prompt of a grouped-query model
        _case("prefill_gqa_long", "prefill", "gqa32", "gqa_long", layers=2, batch=1, ctx_lo=32768, ctx_hi=32768),
        # 8 new tokens of every sequence in one call (speculative verification)
        _case("verify_160m", "separate", "mha12", "160m", layers=4, batch=32, ctx_lo=2048, ctx_hi=2048, chunk=8),
        # a mode per query head (the paper's default granularity)
        _case("heads_160m", "heads", "mha12", "160m", layers=12, batch=32, ctx_lo=2048, ctx_hi=2048, steps=2),
        # steps driven by router logits: decisions and cost, append, attention
        _case("routed_160m", "routed", "mha12", "160m", layers=12, batch=32, ctx_lo=2048, ctx_hi=2048, steps=2),
        # decisions and cost of a whole batch of prompts in one call
        _case("decisions_4m", "decisions", "mha12", "160m", batch=1 << 22, ctx_lo=1, ctx_hi=4096),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["decode"] * 6 + ["prefill"] * 2 + ["separate", "heads", "routed", "decisions", "generate"])
    if kind == "decisions":
        c = _case("", kind, rng.choice(["mha12", "mha32", "gqa32"]), "160m", batch=_log(rng, 64, 1 << 22),
                  ctx_lo=1, ctx_hi=_log(rng, 64, 32768))
        del c["name"]
        return c
    shape = rng.choice(["mha12", "mha12", "mha32", "mha32", "gqa32", "gqa32", "gqa4", "mha8w", "gqa8w", "gqa12"])
    hq, hkv, d, _ = SHAPES[shape]
    mix = rng.choice(["160m", "160m", "1p3b", "gqa_long", "tiny"])
    page = rng.choice([32, 32, 32, 16, 64])
    window = rng.choice([32, 256, 512, 1024])
    if kind == "generate":
        hi = _log(rng, 20, 130)
        c = _case("", kind, shape, mix, page=page, batch=_log(rng, 1, 8), ctx_lo=max(1, hi // 4), ctx_hi=hi,
                  window=window)
        del c["name"]
        return c
    steps, chunk = rng.choice([1, 2, 3]), 1
    most = 256
    if kind == "separate":
        steps, chunk = 1, rng.choice([1, 2, 3, 4, 5, 8])
        most = 64
    elif kind == "prefill":
        most = 64
    batch = _log(rng, 1, most)
    # tokens of a layer, so that no draw costs more than the largest listed case
    room = 256 * 4096 * 2048 // (hkv * d) * 2 // max(steps, 2)
    room //= {"separate": 2 * chunk, "heads": 4}.get(kind, 1) * (4 if hq != hkv or d > 64 else 1)
    top = min(32768 if hq != hkv else 8192, max(64, room // batch))
    if kind == "prefill":
        top = min(top, max(64, 32768 // batch))
    hi = _log(rng, 48, top)
    lo = rng.choice([hi, max(16, hi // 8), max(16, hi // 2)])
    layers = 24 if batch * hi <= 8192 else 12 if batch * hi <= 65536 else 3
    if kind == "prefill":
        layers = rng.choice([1, 2, 4])
    c = _case("", kind, shape, mix, page=page, layers=layers, batch=batch, ctx_lo=lo, ctx_hi=hi, window=window,
              steps=steps, chunk=chunk)
    del c["name"]
    return c


# ------------------------------------------------------------------------- inputs --

def _gen(*key):
    s = 0x9E3779B9
    for k in key:
        s = (s * 6364136223846793005 + int(k) + 1442695040888963407) % (1 << 62)
    g = torch.Generator(device="cuda")
    g.manual_seed(s)
    return g


def _pick(p, shape, g):
    """Indices drawn with probabilities p."""
    edges = torch.tensor(p, device="cuda", dtype=torch.float32).cumsum(0)[:-1].contiguous()
    return torch.bucketize(torch.rand(shape, generator=g, device="cuda"), edges, right=True)


def _contexts(case, seed):
    lo, hi, n = case["ctx_lo"], case["ctx_hi"], case["batch"]
    if case["kind"] == "generate":  # from the shortest to the longest
        return [hi - (hi - lo) * (n - 1 - i) // max(1, n - 1) for i in range(n)]
    if lo == hi:
        return [hi] * n
    return torch.randint(lo, hi + 1, (n,), generator=_gen(seed, 1), device="cuda").tolist()


def _grow(case):
    """Tokens each sequence gets after its prompt."""
    return case["steps"] * case["chunk"] if case["kind"] in ("decode", "separate", "heads", "routed") else 0


def _layer(case, seed, layer, ctx):
    """One layer's tokens, sequence after sequence (a sequence's prompt, then the tokens
    that the steps add): widths, modes, K, V, Q rows."""
    hq, hkv, d, _ = SHAPES[case["shape"]]
    pb, pm, outliers, gap = MIXES[case["mix"]]
    n = sum(ctx) + len(ctx) * _grow(case)
    g = _gen(seed, 2, layer)
    bits = torch.tensor(BITS, device="cuda", dtype=torch.uint8)[_pick(pb, (n,), g)]
    if gap:
        lens = torch.randint(gap[0], gap[1] + 1, (n // gap[0] + 1,), generator=g, device="cuda")
        at = torch.cat([lens.new_zeros(1), lens.cumsum(0)])
        bits[at[at < n]] = 16
    heads = (hq,) if case["kind"] == "heads" else ()
    modes = _pick(pm, (n,) + heads, g).to(torch.uint8)
    k = torch.randn((n, hkv, d), generator=g, device="cuda", dtype=torch.bfloat16)
    v = torch.randn((n, hkv, d), generator=g, device="cuda", dtype=torch.bfloat16)
    if outliers:
        ch = torch.randperm(hkv * d, generator=g, device="cuda")[: math.ceil(0.01 * hkv * d)]
        k.view(n, -1)[:, ch] *= 8
        v.view(n, -1)[:, ch] *= 8
    return bits, modes, k, v


def _queries(case, seed, layer, step, n):
    hq, _, d, _ = SHAPES[case["shape"]]
    return torch.randn((n, hq, d), generator=_gen(seed, 3, layer, step), device="cuda", dtype=torch.bfloat16)


def _logits(options, picked, g):
    """Router logits whose arg max is `picked`."""
    z = torch.rand((picked.numel(), options), generator=g, device="cuda") - 2.0
    z[torch.arange(picked.numel(), device="cuda"), picked.long()] = 1.0
    return z


def _starts(ctx, extra):
    s, out = 0, []
    for c in ctx:
        out.append(s)
        s += c + extra
    return out


def _steps(case, ctx):
    """Per step: the (sequence, position) entries, in call order."""
    if case["kind"] == "generate":
        return [[(s, p) for s in range(len(ctx)) if p < ctx[s]] for p in range(max(ctx))]
    C = case["chunk"]
    return [[(s, ctx[s] + i * C + j) for s in range(len(ctx)) for j in range(C)] for i in range(case["steps"])]


def _i32(x):
    return torch.tensor(x, dtype=torch.int32, device="cuda")


# ------------------------------------------------------------------------ prepare --

def prepare(case, seed):
    if case["kind"] == "decisions":
        return _prepare_decisions(case, seed)
    hq, hkv, d, G = SHAPES[case["shape"]]
    kind, L, P, B = case["kind"], case["layers"], case["page"], case["batch"]
    ctx = _contexts(case, seed)
    extra = _grow(case)
    maxctx = case["ctx_hi"] + extra + 1
    pb = MIXES[case["mix"]][0]
    gap = MIXES[case["mix"]][3]
    # room for every sequence's pages in every class: the expected share and some more
    total = B * (case["ctx_hi"] + extra)
    caps = []
    for b, p in zip(BITS, pb):
        p += 1 / gap[0] if gap and b == 16 else 0
        caps.append(int(L * (total * min(1.0, 1.1 * p) / P + 8 * math.sqrt(total) / P + 2 * B + 8)))
    n_call = B * case["chunk"]
    cache = trr.Cache(L, B, hq, hkv, d, G, P, maxctx, caps, max_append=1024, max_queries=max(64, n_call),
                      head_modes=1 if kind == "heads" else 0, zero_pool=True)
    starts = _starts(ctx, extra)
    prompt = ctx if kind != "generate" else [0] * B
    seq_ids = torch.repeat_interleave(torch.arange(B, device="cuda"), torch.tensor(prompt, device="cuda"))
    if seq_ids.numel():
        first = torch.tensor([sum(prompt[:s]) for s in range(B)], device="cuda")
        pos = torch.arange(seq_ids.numel(), device="cuda") - first[seq_ids]
        rows = torch.tensor(starts, device="cuda")[seq_ids] + pos
        seq_ids, pos = seq_ids.to(torch.int32), pos.to(torch.int32)
    steps = _steps(case, ctx) if kind != "prefill" else []
    index = [(_i32([s for s, _ in e]), _i32([p for _, p in e]),
              torch.tensor([starts[s] + p for s, p in e], device="cuda")) for e in steps]
    calls, work = [], [[] for _ in steps]
    for l in range(L):
        bits, modes, k, v = _layer(case, seed, l, ctx)
        chunks = []
        for e0 in range(0, seq_ids.numel(), 1024):
            r = rows[e0:e0 + 1024]
            chunks.append((l, seq_ids[e0:e0 + 1024].contiguous(), pos[e0:e0 + 1024].contiguous(), k[r], v[r],
                           bits[r], modes[r]))
            if kind != "prefill":
                cache.append(*chunks.pop())
        calls += chunks
        for i, (ids, ps, r) in enumerate(index):
            w = {"layer": l, "ids": ids, "pos": ps, "k": k[r], "v": v[r], "bits": bits[r], "modes": modes[r],
                 "q": _queries(case, seed, l, i, ids.numel())}
            if kind == "routed":
                g = _gen(seed, 4, l, i)
                w["mode_logits"] = _logits(3, w["modes"], g)
                w["bit_logits"] = _logits(4, torch.log2(w["bits"].float()).round().to(torch.int64) - 1, g)
            work[i].append(w)
    torch.cuda.synchronize()
    if cache.status() != 0:
        raise RuntimeError("the prompts do not fit the cache")
    state = {"kind": kind, "cache": cache, "calls": calls}
    regions = [cache.region(r) for r in ("last_pos", "ntok", "presence", "page_table", "page_first", "page_last",
                                          "next_page", "pool2", "pool4", "pool8", "pool16")]
    if kind == "prefill":
        state["outputs"] = regions
        return state
    rows = torch.empty(sum(L * ids.numel() * hq * d for ids, _, _ in index), dtype=torch.bfloat16, device="cuda")
    outs, at = [], 0
    for ids, _, _ in index:
        outs.append(rows[at:at + L * ids.numel() * hq * d].view(L, ids.numel(), hq, d))
        at += outs[-1].numel()
    totals = torch.zeros(4, dtype=torch.int64, device="cuda")
    if kind != "generate":
        # the cache's bookkeeping (everything before its per-call scratch) as the prompts left it
        last = cache.region("page_last")
        end = last.data_ptr() + last.numel() - cache.pool.data_ptr()
        end = (end + 255) // 256 * 256 + 16 * L * B
        state["book"] = cache.pool[:end]
        state["prompt_book"] = state["book"].clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for i, layers in enumerate(work):
            for w in layers:
                _enqueue(case, cache, w, outs[i][w["layer"]], totals)
    state.update(graph=graph, work=work, totals=totals, outputs=[rows] + regions)
    if kind == "routed":
        state["outputs"] = state["outputs"] + [totals]
    return state


def _enqueue(case, cache, w, out, totals):
    """One layer's calls of one step."""
    l, ids, pos, win = w["layer"], w["ids"], w["pos"], case["window"]
    hq, hkv, d, _ = SHAPES[case["shape"]]
    if case["kind"] in ("decode", "generate"):
        cache.decode_step(l, ids, pos, w["k"], w["v"], w["bits"], w["modes"], w["q"], window_scalar=win, out=out)
    elif case["kind"] == "routed":
        trr.trr_route_decisions(w["mode_logits"], w["bit_logits"], pos, win, hq, d, hkv, totals=totals)
        cache.append_routed(l, ids, pos, w["k"], w["v"], w["bit_logits"], w["mode_logits"])
        cache.decode_attn_routed(l, ids, pos, w["q"], w["mode_logits"], window_scalar=win, out=out)
    else:
        cache.append(l, ids, pos, w["k"], w["v"], w["bits"], w["modes"])
        cache.decode_attn(l, ids, pos, w["q"], w["modes"], window_scalar=win, out=out)


def _prepare_decisions(case, seed):
    n = case["batch"]
    g = _gen(seed, 5)
    dev = {"device": "cuda"}
    return {"kind": "decisions", "case": case,
            "mode_logits": torch.randn((n, 3), generator=g, **dev), "bit_logits": torch.randn((n, 4), generator=g, **dev),
            "pos": torch.randint(case["ctx_lo"] - 1, case["ctx_hi"], (n,), generator=g, dtype=torch.int32, **dev),
            "modes": torch.empty(n, dtype=torch.uint8, **dev), "bits": torch.empty(n, dtype=torch.uint8, **dev),
            "flops": torch.empty(n, dtype=torch.int64, **dev), "kv": torch.empty(n, dtype=torch.int64, **dev),
            "totals": torch.zeros(4, dtype=torch.int64, **dev)}


# ---------------------------------------------------------------------------- run --

def run(state):
    if state["kind"] == "decisions":
        s, c = state, state["case"]
        hq, hkv, d, _ = SHAPES[c["shape"]]
        s["totals"].zero_()
        trr.trr_route_decisions(s["mode_logits"], s["bit_logits"], s["pos"], c["window"], hq, d, hkv,
                                modes=s["modes"], bits=s["bits"], attn_flops=s["flops"], kv_bits=s["kv"],
                                totals=s["totals"])
        return [s["modes"], s["bits"], s["flops"], s["kv"], s["totals"]]
    cache = state["cache"]
    if state["kind"] == "prefill":
        cache.reset()
        for call in state["calls"]:
            cache.append(*call)
        return state["outputs"]
    if state["kind"] == "generate":
        cache.reset()
    else:
        state["book"].copy_(state["prompt_book"])
    if state["kind"] == "routed":
        state["totals"].zero_()
    state["graph"].replay()
    return state["outputs"]


# --------------------------------------------------------------------------- work --

def _token_bytes(b, d, G):
    """K and V of one token and KV head, as stored."""
    return 4 * d if b == 16 else 2 * (d * b // 8) + 8 * (d // G)


def work(case):
    """Expected over the case's mix: stored keys in range (their codes, scales and
    positions) read once a call and sequence, new rows read and stored, Q and O rows."""
    hq, hkv, d, G = SHAPES[case["shape"]]
    pb, pm, _, gap = MIXES[case["mix"]]
    if case["kind"] == "decisions":
        return {"bytes": 50 * case["batch"], "flops": 0}
    if gap:
        f = 2.0 / (gap[0] + gap[1])
        pb = [p * (1 - f) for p in pb[:3]] + [pb[3] * (1 - f) + f]
    per_head = sum(p * _token_bytes(b, d, G) for b, p in zip(BITS, pb))
    skip, local, full = pm
    B, L, C, w = case["batch"], case["layers"], case["chunk"], case["window"]
    mean = (case["ctx_lo"] + case["ctx_hi"]) / 2
    if case["kind"] == "prefill":
        n = B * mean * L
        return {"bytes": n * hkv * d * 4 * (1 - skip) + n * (1 - skip) * (hkv * per_head + 4), "flops": 0}
    if case["kind"] == "generate":
        n, length = B * mean, mean / 2
        steps = 1
    else:
        n, length = B * C, mean
        steps = case["steps"]
    if case["kind"] == "heads":
        stored, keys = 1 - skip ** hq, (full * length + local * min(w, length)) * (1 - skip) * hkv
        groups = 1
    else:
        # the queries of a sequence read its pages once a call
        stored, groups = 1 - skip, C
        reads_full, reads_any = 1 - (1 - full) ** C, 1 - skip ** C
        keys = (reads_full * length + (reads_any - reads_full) * min(w + C, length)) * (1 - skip) * hkv / C
    attended = (full * length + local * min(w, length)) * (1 - skip) * hq
    nbytes = n * (keys * (per_head + 4 / hkv) + stored * hkv * (4 * d + per_head) + hq * d * 4)
    return {"bytes": nbytes * steps * L, "flops": n * attended * 4 * d * steps * L}


# -------------------------------------------------------------------------- exact --

def _stored(x, bits, G):
    """K or V rows [n][heads][d] as the cache stores them (Eq. 4 at each token's width),
    in 64 bits."""
    out = x.double()
    for b in (2, 4, 8):
        at = (bits == b).nonzero().flatten()
        if not at.numel():
            continue
        g = x[at].float().unflatten(-1, (-1, G))
        lo, hi = g.amin(-1, keepdim=True), g.amax(-1, keepdim=True)
        z = lo.half().double()
        s = ((hi - lo) / float((1 << b) - 1)).half().double()
        c = torch.where(s > 0, (g.double() - z) / torch.where(s > 0, s, torch.ones_like(s)), torch.zeros_like(z))
        c = c.round().clamp_(0, (1 << b) - 1)
        out[at] = (z + c * s).flatten(-2)
    return out


def exact(case, seed):
    if case["kind"] in ("decisions", "prefill"):
        return None
    hq, hkv, d, G = SHAPES[case["shape"]]
    ctx = _contexts(case, seed)
    extra = _grow(case)
    starts = _starts(ctx, extra)
    steps = _steps(case, ctx)
    L, w, grp = case["layers"], case["window"], hq // hkv
    outs = [torch.zeros((L, len(e), hq, d), dtype=torch.float64, device="cuda") for e in steps]
    by_seq = [[] for _ in ctx]
    for i, e in enumerate(steps):
        for j, (s, p) in enumerate(e):
            by_seq[s].append((i, j, p))
    for l in range(L):
        bits, modes, k, v = _layer(case, seed, l, ctx)
        qs = [_queries(case, seed, l, i, len(e)) for i, e in enumerate(steps)]
        # every token's mode per query head
        per_head = modes if modes.dim() == 2 else modes[:, None].expand(-1, hq)
        for s, start in enumerate(starts):
            n = ctx[s] + extra
            m = per_head[start:start + n]
            asked = m[torch.tensor([p for _, _, p in by_seq[s]], device="cuda")].tolist()
            if not any(map(any, asked)):
                continue
            low = 0
            if not any(FULL in a for a in asked):
                low = max(0, min(p for _, _, p in by_seq[s]) - w + 1)
            at = slice(start + low, start + n)
            K, V = _stored(k[at], bits[at], G), _stored(v[at], bits[at], G)
            # KV head j of a token is there when a query head reading it does not skip
            there = (m[low:].unflatten(1, (hkv, grp)) != SKIP).any(-1)
            place = torch.arange(low, n, device="cuda")
            for (i, j, p), a in zip(by_seq[s], asked):
                if not any(a):
                    continue
                upto = p + 1 - low
                mine = torch.tensor(a, device="cuda")
                first = torch.where(mine == FULL, 0, p - w + 1)
                q = qs[i][j].double().unflatten(0, (hkv, grp))
                score = torch.einsum("hgd,nhd->hgn", q, K[:upto]).flatten(0, 1) / math.sqrt(d)
                ok = (place[None, :upto] >= first[:, None]) & (mine != SKIP)[:, None]
                ok &= there[:upto].T.repeat_interleave(grp, 0)
                score = score.masked_fill(~ok, -math.inf)
                top = score.amax(-1, keepdim=True)
                e = torch.exp(score - torch.where(torch.isfinite(top), top, torch.zeros_like(top)))
                o = torch.einsum("hgn,nhd->hgd", e.unflatten(0, (hkv, grp)), V[:upto]).flatten(0, 1)
                total = e.sum(-1, keepdim=True)
                outs[i][l, j] = torch.where(total > 0, o / total.clamp_min(1e-300), torch.zeros_like(o))
    return [torch.cat([o.flatten() for o in outs])] + [None] * (12 if case["kind"] == "routed" else 11)
