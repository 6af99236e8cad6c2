"""Performance cases of the VarRate codec: what a serving program asks of the library.

A case names one operation and its sizes. The operations, each through the public entry points of
``paper_2607_15498_gb300.varrate``:

* ``prefill``   varrate_encode of a prompt's cache, then the first decode call of every layer. The
                outputs are the salience, the ranks and the attention of that first token: which
                slot of the packed cache a token takes depends on every rank before it, so a rank
                that falls the other way at a tie moves the slots of all later tokens, and the
                attention is where the packed coefficients of two correct runs can be compared.
* ``pack``      varrate_allocate and varrate_pack on a given salience; all tables and coefficients.
* ``decode``    one decode step through every layer, replayed from a CUDA graph as a serving loop
                that captures its step does (fp32 cases issue the calls directly).
* ``window``    varrate_decode_window of n_q new tokens on every layer (speculative or chunked).
* ``quantize``  varrate_quantize of a packed cache.
* ``decode_q``  one decode step on the quantized cache through every layer, from a CUDA graph.
* ``search``    varrate_anchor_search; ``residual``  varrate_anchor_residual (joint codec).

Keys and values are low-rank plus noise or have a decaying spectrum in a random orthonormal frame;
the basis handed to the codec is that frame, as an offline calibration would find it. ``outliers``
is the share of tokens with 8x keys (what the salience has to pick out); where the salience is an
input it is log-normal of width ``spread`` (0.15: nearly flat, ranks within a few units of each
other; 1.0: heavy-tailed, ranks from r_min to head_dim).
"""
import math

import torch

from paper_2607_15498_gb300 import varrate as V

D = 128
OPS = ("prefill", "pack", "decode", "window", "quantize", "decode_q", "search", "residual")


def _case(op, **kw):
    c = {"op": op, "layers": 1, "kv_heads": 8, "group": 4, "n": 32768, "batch": 1, "budget": 0.2,
         "r_min": 16, "window": 32, "dtype": "bf16", "spectrum": "lowrank", "outliers": 0.0,
         "spread": 0.15, "uniform": False, "tail": 0, "n_q": 0, "bits": 0, "stride": 0, "c": 0}
    c.update(kw)
    return c


def listed():
    return [
        # a short prompt of one small fp32 layer: every kernel is small, latency and launches count
        dict(_case("prefill", kv_heads=1, n=2048, dtype="f32", spectrum="inv", outliers=0.05), name="prefill_tiny_f32"),
        # a model that prefills layer by layer encodes one layer's 32k cache at a time
        dict(_case("prefill", outliers=0.05), name="prefill_layer_32k"),
        # the whole 32-layer cache of one 32k prompt in one call: bandwidth
        dict(_case("prefill", layers=32), name="prefill_stack_32k"),
        # a caller with a salience of its own (another window, another method) packs with it
        dict(_case("pack", layers=4, kv_heads=4, group=7, n=32749, budget=0.3, spectrum="pow", spread=1.0), name="pack_own_salience"),
        # one decode step of eight sequences: the serving batch, four layers of it
        dict(_case("decode", layers=4, batch=8), name="decode_batch8_32k"),
        # one decode step of a single sequence with GQA group 7 through 28 layers: latency
        dict(_case("decode", layers=28, kv_heads=4, group=7, spectrum="pow", spread=1.0), name="decode_single_32k"),
        # long-context reuse: 131072 tokens, 97 exact tokens appended since the encode
        dict(_case("decode", layers=8, n=131072, tail=97, spread=0.5), name="decode_long_tail"),
        # 32 new tokens at once (the observation window of a new query batch) on the long cache
        dict(_case("window", layers=2, n=131072, tail=32, n_q=32), name="window_32_long"),
        # the packed cache of eight sequences in 8-bit form, once after each encode
        dict(_case("quantize", layers=2, batch=8, bits=8), name="quantize_8bit"),
        # the serving batch on a 4-bit cache
        dict(_case("decode_q", layers=4, batch=8, bits=4), name="decode_q4_batch8"),
        # the joint codec on one 32k layer: the nearest anchors, then the residuals
        dict(_case("search", stride=16, c=4), name="anchor_search_32k"),
        dict(_case("residual", layers=2, n=32768, stride=16, c=4), name="anchor_residual_32k"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(OPS)
    G, grp = rng.randint(1, 8), rng.randint(1, 8)
    n = _log(rng, 600, 131072)
    f32 = op in ("prefill", "pack", "decode") and rng.random() < 0.2
    room = (1 << 19) if f32 else (1 << 20) if op in ("search",) else (1 << 22)   # K/V rows in all
    if op == "search":
        n = min(n, 40000)
    if f32:
        n = min(n, 9000)
    batch = rng.randint(1, 8) if op in ("decode", "decode_q", "quantize") else rng.randint(1, 2)
    batch = max(1, min(batch, room // (n * G)))
    layers = max(1, min(rng.randint(1, 12), room // (n * G * batch)))
    window = rng.choice([w for w in (8, 16, 17, 32, 48, 64) if w * grp <= 256])
    kw = dict(layers=layers, kv_heads=G, group=grp, n=n, batch=batch, window=window,
              budget=round(rng.uniform(0.15, 0.6), 3), r_min=rng.choice([1, 8, 16, 16, 24]),
              dtype="f32" if f32 else "bf16", spectrum=rng.choice(["lowrank", "pow", "inv"]),
              spread=round(rng.uniform(0.1, 1.2), 2), outliers=rng.choice([0.0, 0.02, 0.05]))
    if op in ("prefill", "pack"):
        kw["uniform"] = rng.random() < 0.1
    if op in ("decode", "decode_q"):
        kw["tail"] = rng.choice([0, 0, 1, _log(rng, 2, 256), rng.randint(257, 600)])
    if op == "window":
        kw["n_q"] = rng.randint(1, 128 // grp)
        kw["tail"] = kw["n_q"] + rng.choice([0, rng.randint(1, 300)])
    if op in ("quantize", "decode_q"):
        kw["bits"] = rng.choice([4, 8])
    if op in ("search", "residual"):
        kw["stride"], kw["c"] = rng.choice([5, 8, 16, 16, 32, 33]), rng.randint(1, 8)
        if op == "search":   # n^2 G / stride distances: no more than the listed search's work
            kw["stride"] = max(kw["stride"], -(-n * n * G * batch * layers // (1 << 29)))
    return _case(op, **kw)


# ------------------------------------------------------------------------------------ inputs

def _gen(seed, salt):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed * 1000003 + salt)
    return g


def _dt(c):
    return torch.float32 if c["dtype"] == "f32" else torch.bfloat16


def _frames(c, seed):
    """Orthonormal frames [L][G][2][d][d] (fp64), column i = direction i."""
    a = torch.randn((c["layers"], c["kv_heads"], 2, D, D), generator=_gen(seed, 1), device="cuda")
    return torch.linalg.qr(a.double().cpu())[0].cuda()


def _bases(c, F):
    b = F.transpose(-1, -2).to(_dt(c))
    return b[:, :, 0].contiguous(), b[:, :, 1].contiguous()


def _kv(c, seed, F):
    """Keys and values [B][L][G][N][d]."""
    i = torch.arange(1, D + 1, device="cuda", dtype=torch.float32)
    sig = {"lowrank": (i <= 40).float(), "pow": i ** -0.7, "inv": 1.0 / i}[c["spectrum"]]
    noise = 0.05 if c["spectrum"] == "lowrank" else 0.0
    sig = sig * math.sqrt((1.0 - noise * noise) * D / float((sig * sig).sum()))
    B, L, G, n = c["batch"], c["layers"], c["kv_heads"], c["n"]
    out = [torch.empty((B, L, G, n, D), dtype=_dt(c), device="cuda") for _ in range(2)]
    g = _gen(seed, 2)
    local = c["op"] in ("search", "residual")   # neighbouring tokens are alike: what anchors are for
    # keys of the outlier tokens; the last w tokens are the exact set
    hot = torch.rand((B, L, n), generator=g, device="cuda") < c["outliers"]
    hot[:, :, n - c["window"]:] = False
    for b in range(B):
        for l in range(L):
            for kv in range(2):
                z = torch.randn((G, n, D), generator=g, device="cuda")
                if local:
                    seg = torch.randn((G, (n + 63) // 64, D), generator=g, device="cuda")
                    z = 0.8 * seg.repeat_interleave(64, dim=1)[:, :n] + 0.6 * z
                x = torch.matmul(z * sig, F[l, :, kv].float().transpose(-1, -2))
                if noise:
                    x += noise * torch.randn(x.shape, generator=g, device="cuda")
                if kv == 0 and c["outliers"] and not local:
                    x *= torch.where(hot[b, l], 8.0, 1.0)[None, :, None]
                out[kv][b, l] = x.to(_dt(c))
    return out


def _salience(c, seed):
    z = torch.randn((c["batch"], c["layers"], c["n"] - c["window"]), generator=_gen(seed, 3), device="cuda")
    return torch.exp(c["spread"] * z) / c["n"]


def _queries(c, seed, n_q, salt):
    H = c["kv_heads"] * c["group"]
    shape = (c["layers"], c["batch"], n_q, H, D)
    return torch.randn(shape, generator=_gen(seed, salt), device="cuda").to(_dt(c))


def _tail(c, seed):
    shape = (2, c["layers"], c["batch"], c["kv_heads"], c["tail"], D)
    return torch.randn(shape, generator=_gen(seed, 5), device="cuda").to(_dt(c))


def _lists(c, seed):
    """Anchor lists as the search gives them: the anchor before the token and others, distinct."""
    B, L, n = c["batch"], c["layers"], c["n"]
    n_a = -(-n // c["stride"])
    k = min(c["c"], n_a)
    near = torch.arange(n, device="cuda") // c["stride"]
    step = max(1, n_a // max(1, k))
    off = torch.randint(0, step, (B, L, n, k), generator=_gen(seed, 6), device="cuda") + step * torch.arange(k, device="cuda")
    off[..., 0] = 0
    idx = torch.full((B, L, n, c["c"]), -1, dtype=torch.int32, device="cuda")
    idx[..., :k] = ((near[:, None] + off) % n_a).int()
    return idx


def _cfg(c):
    return V.make_config(c["layers"], c["kv_heads"], c["group"], c["n"], batch=c["batch"],
                         budget_frac=c["budget"], r_min=c["r_min"], window=c["window"],
                         dtype=V.F32 if c["dtype"] == "f32" else V.BF16,
                         mode=V.UNIFORM if c["uniform"] else V.SALIENCE)


def _workspace(nbytes):
    return torch.zeros(max(nbytes, 256), dtype=torch.uint8, device="cuda")


class _State:
    pass


def prepare(case, seed):
    c, s = case, _State()
    s.c, s.cfg, s.graph = c, _cfg(c), None
    cfg = s.cfg
    F = _frames(c, seed)
    s.bk, s.bv = _bases(c, F)
    s.status = torch.zeros(1, dtype=torch.int32, device="cuda")
    s.k, s.v = _kv(c, seed, F)
    B, L, H, n = c["batch"], c["layers"], c["kv_heads"] * c["group"], c["n"]
    op = c["op"]
    if op == "search":
        s.idx = torch.empty((B, L, n, c["c"]), dtype=torch.int32, device="cuda")
        s.dist = torch.empty((B, L, n, c["c"]), dtype=torch.float32, device="cuda")
        s.ws = _workspace(V.varrate_anchor_search_ws_bytes(cfg, c["stride"]))
        return s
    if op == "residual":
        s.idx = _lists(c, seed)
        s.e = torch.empty((B, L, n, 2 * c["kv_heads"] * D), dtype=torch.bfloat16, device="cuda")
        return s
    s.packed = V.PackedCache.allocate(cfg)
    s.packed.coef.zero_()      # elements past the last bucket are never written
    s.q = _queries(c, seed, max(1, c["n_q"]), 4)
    s.tk, s.tv = _tail(c, seed) if c["tail"] else (None, None)
    s.out = torch.empty_like(s.q)
    if op == "prefill":
        s.qw = _queries(c, seed, c["window"], 7).permute(1, 0, 2, 3, 4).contiguous()
        s.sal = torch.empty((B, L, n - c["window"]), dtype=torch.float32, device="cuda")
        s.ws_enc = V.workspace(cfg, V.CALL_ENCODE)
        s.ws = V.workspace(cfg, V.CALL_DECODE)
        return s
    s.sal = _salience(c, seed)
    s.realized = torch.zeros((B, L), dtype=torch.int64, device="cuda")
    s.ws_pack = V.workspace(cfg, V.CALL_PACK)
    if op == "pack":
        return s
    _pack(s)
    torch.cuda.synchronize()
    s.k = s.v = None
    if op in ("quantize", "decode_q"):
        s.qpacked = V.QPackedCache.allocate(cfg, s.packed, c["bits"])
        if op == "quantize":
            return s
        V.check(V.varrate_quantize(cfg, s.packed, s.qpacked, s.status), "varrate_quantize")
    if op == "window":
        s.ws = V.workspace(cfg, V.CALL_DECODE_WINDOW)
        return s
    s.ws = V.workspace(cfg, V.CALL_DECODE_Q if op == "decode_q" else V.CALL_DECODE)
    if c["dtype"] == "bf16":
        _step(s)               # the first calls on a device and a workspace come before the capture
        torch.cuda.synchronize()
        s.graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s.graph):
            _step(s)
    return s


def _pack(s):
    V.check(V.varrate_allocate(s.cfg, s.sal, s.packed.ranks, s.realized, s.status), "varrate_allocate")
    V.check(V.varrate_pack(s.cfg, s.k, s.v, s.bk, s.bv, s.packed, s.status, s.ws_pack), "varrate_pack")


def _step(s):
    """One decode step: a call for each layer."""
    c = s.c
    for l in range(c["layers"]):
        tk, tv = (s.tk[l], s.tv[l]) if c["tail"] else (None, None)
        if c["op"] == "decode_q":
            V.check(V.varrate_decode_attn_q(s.cfg, s.qpacked, s.bk, s.bv, s.q[l], l, tk, tv, c["tail"],
                                            s.out[l], s.status, s.ws), "varrate_decode_attn_q")
        else:
            V.check(V.varrate_decode_attn(s.cfg, s.packed, s.bk, s.bv, s.q[l], l, tk, tv, c["tail"],
                                          s.out[l], s.status, s.ws), "varrate_decode_attn")


def run(state):
    s, c = state, state.c
    op = c["op"]
    if op == "prefill":
        V.check(V.varrate_encode(s.cfg, s.qw, s.k, s.v, s.bk, s.bv, s.sal, s.packed, None, s.status,
                                 s.ws_enc), "varrate_encode")
        _step(s)
        return {"salience": s.sal, "ranks": s.packed.ranks, "attention": s.out, "status": s.status}
    if op == "pack":
        _pack(s)
        p = s.packed
        return {"ranks": p.ranks, "realized": s.realized, "bucket_count": p.bucket_count,
                "bucket_base": p.bucket_base, "perm": p.perm, "pos": p.pos, "coef": p.coef,
                "status": s.status}
    if op == "quantize":
        V.check(V.varrate_quantize(s.cfg, s.packed, s.qpacked, s.status), "varrate_quantize")
        return {"data": s.qpacked.data, "qbase": s.qpacked.qbase, "status": s.status}
    if op == "search":
        V.check(V.varrate_anchor_search(s.cfg, s.k, s.v, c["stride"], c["c"], s.idx, s.dist, s.status,
                                        s.ws), "varrate_anchor_search")
        return {"idx": s.idx, "dist": s.dist, "status": s.status}
    if op == "residual":
        V.check(V.varrate_anchor_residual(s.cfg, s.k, s.v, c["stride"], c["c"], s.idx, s.e, s.status),
                "varrate_anchor_residual")
        return {"residual": s.e, "status": s.status}
    if op == "window":
        for l in range(c["layers"]):
            V.check(V.varrate_decode_window(s.cfg, s.packed, s.bk, s.bv, s.q[l], c["n_q"], l, s.tk[l],
                                            s.tv[l], c["tail"], s.out[l], s.status, s.ws),
                    "varrate_decode_window")
        return {"attention": s.out, "status": s.status}
    if s.graph is not None:
        s.graph.replay()
    else:
        _step(s)
    return {"attention": s.out, "status": s.status}


# ------------------------------------------------------------------------- work and tolerance

def _budget(c):
    return math.floor(c["budget"] * (c["n"] * D)) - c["window"] * D


def work(case):
    c = case
    e = 4 if c["dtype"] == "f32" else 2
    B, L, G, n, w = c["batch"], c["layers"], c["kv_heads"], c["n"], c["window"]
    H = G * c["group"]
    kv = 2 * B * L * G * n * D * e                                   # K and V
    coded = min(max(_budget(c), c["r_min"] * (n - w)), D * (n - w))
    ranks = B * L * (coded + w * D)                                  # sum of ranks, per head and side
    coef = 2 * G * ranks * e
    nq = max(1, c["n_q"])
    io = 2 * L * G * D * D * e + 2 * L * B * nq * H * D * e          # bases, queries and outputs
    tail = 2 * L * B * G * c["tail"] * D * e
    # scores and values on the coefficients, for each query head
    attn = 4 * nq * c["group"] * G * ranks + 4 * nq * H * L * B * c["tail"] * D + 4 * nq * L * B * H * D * D
    project = 2 * 2 * G * ranks * D
    tables = B * L * n * (1 + 4 + 4)                                 # ranks, perm, pos
    op = c["op"]
    if op == "prefill":
        sal = 2 * B * L * H * w * n * D
        return {"bytes": kv + 2 * coef + io + tables + 4 * B * L * (n - w) + B * L * w * H * D * e,
                "flops": sal + project + attn}
    if op == "pack":
        return {"bytes": kv + coef + 2 * L * G * D * D * e + tables + 4 * B * L * (n - w), "flops": project}
    if op == "quantize":
        q = 2 * G * ranks * (c["bits"] + 1) // 8
        return {"bytes": coef + q, "flops": 8 * G * ranks}
    if op == "search":
        n_a = -(-n // c["stride"])
        return {"bytes": kv + B * L * n * c["c"] * 8, "flops": 2 * B * L * n * n_a * 2 * G * D}
    if op == "residual":
        return {"bytes": 2 * kv + B * L * n * c["c"] * 4, "flops": B * L * n * 2 * G * D * (c["c"] + 2)}
    if op == "decode_q":
        return {"bytes": 2 * G * ranks * (c["bits"] + 1) // 8 + io + tail, "flops": attn}
    return {"bytes": coef + io + tail, "flops": attn}


def tolerance(case):
    op = case["op"]
    if op == "quantize":
        return "exact"          # codes and group parameters are a function of the stored bits
    if op == "search":          # fp32 sums; two anchors closer than their rounding change places
        return {"rel": 2e-5, "max": 1e-3, "differ": 2e-3}
    if op == "residual":        # a bf16 result of fp32 sums
        return {"rel": 1e-3, "max": 2e-2}
    if case["dtype"] == "f32":
        return {"rel": 2e-5, "max": 1e-3, "differ": 2e-3 if op == "prefill" else 0.0}
    if op == "prefill":         # ranks at a tie follow the last bits of the salience
        return {"rel": 2e-2, "max": 2e-1, "differ": 2e-3}
    if op == "pack":            # bf16 storage of fp32 sums
        return {"rel": 1e-3, "max": 2e-2}
    return {"rel": 1e-2, "max": 1e-1}


# --------------------------------------------------------------------------------- in 64 bits

def _ranks(c, sal):
    """Ranks [n] of one (sequence, layer) from its fp32 salience, every operation in IEEE fp32."""
    n, w = c["n"], c["window"]
    bc, nc = _budget(c), n - w
    full = torch.full((n,), D, dtype=torch.int64, device=sal.device)
    if nc == 0 or bc >= D * nc:
        return full
    if c["r_min"] * nc > bc:
        full[:nc] = c["r_min"]
        return full
    mn, mx = sal.min(), sal.max()
    sh = torch.ones_like(sal) if c["uniform"] or not bool(mx > mn) else (sal - mn) / (mx - mn)

    def at(bits):
        lam = torch.tensor(bits, dtype=torch.int32).view(torch.float32).to(sal.device)
        x = torch.mul(sh, lam) + float(c["r_min"])
        return torch.clamp(torch.floor(torch.clamp(x, max=float(D))), min=c["r_min"]).long()
    lo, hi = 0, 0x7F7FFFFF
    if int(at(hi).sum()) <= bc:
        lo = hi
    while hi - lo > 1:
        mid = (lo + hi) // 2
        if int(at(mid).sum()) <= bc:
            lo = mid
        else:
            hi = mid
    full[:nc] = at(lo)
    return full


def _quantized(c, coef, ranks):
    """Coefficients [G][N][d] of one stream kind through group-wise b-bit codes (fp32 steps)."""
    out = torch.zeros_like(coef)
    top = float((1 << c["bits"]) - 1)
    for r in torch.unique(ranks).tolist():
        t = torch.nonzero(ranks == r).flatten()
        m = t.numel()
        x = coef[:, t, :r].float()
        x8 = torch.zeros((x.shape[0], -(-m // 8) * 8, r), device=x.device)
        x8[:, :m] = x
        inf = torch.full((x.shape[0], -(-m // 32) * 32 - x8.shape[1], r), float("inf"), device=x.device)
        lo = torch.cat([x8, inf], 1).view(x.shape[0], -1, 32, r).amin(2)
        hi = torch.cat([x8, -inf], 1).view(x.shape[0], -1, 32, r).amax(2)
        lo = lo.half().float()
        step = torch.clamp((hi - lo) / top, max=65504.0).half().float()
        lo, step = (a.repeat_interleave(32, 1)[:, :m] for a in (lo, step))
        code = torch.where(step > 0, torch.clamp(torch.round((x - lo) / step), 0, top), torch.zeros_like(x))
        out[:, t, :r] = (lo + code * step).to(out.dtype)
    return out


def _attend(c, q, ck, cv, ranks, bk, bv, tk, tv):
    """q [n_q][H][d] -> [n_q][H][d] on coefficients [G][N][d], query i causal over the tail."""
    G, grp, n_q = c["kv_heads"], c["group"], q.shape[0]
    qg = q.view(n_q, G, grp, D).permute(1, 0, 2, 3).reshape(G, n_q * grp, D)
    s = torch.matmul(torch.matmul(qg, bk.transpose(-1, -2)), ck.transpose(-1, -2)) / math.sqrt(D)
    if c["tail"]:
        st = torch.matmul(qg, tk.transpose(-1, -2)) / math.sqrt(D)
        at = torch.arange(c["tail"], device=q.device)
        last = c["tail"] - n_q + torch.arange(n_q, device=q.device).repeat_interleave(grp)
        if c["op"] == "window":
            st = st.masked_fill(at[None, None, :] > last[None, :, None], -math.inf)
        s = torch.cat([s, st], -1)
    p = torch.softmax(s, -1)
    o = torch.matmul(torch.matmul(p[..., :c["n"]], cv), bv)
    if c["tail"]:
        o = o + torch.matmul(p[..., c["n"]:], tv)
    return o.view(G, n_q, grp, D).permute(1, 0, 2, 3).reshape(n_q, G * grp, D)


def exact(case, seed):
    c = case
    if c["op"] == "quantize":
        return None             # bytes, compared bit for bit
    B, L, G, n, w = c["batch"], c["layers"], c["kv_heads"], c["n"], c["window"]
    F = _frames(c, seed)
    bk, bv = (b.double() for b in _bases(c, F))
    k, v = _kv(c, seed, F)
    if c["op"] in ("search", "residual"):
        z = torch.cat([k, v], 2).permute(0, 1, 3, 2, 4).reshape(B, L, n, 2 * G * D)
        if c["op"] == "residual":
            res = torch.empty((B, L, n, 2 * G * D), device="cuda")
            idx = _lists(c, seed).long()
            live = idx >= 0
            for b in range(B):
                for l in range(L):
                    a = z[b, l, ::c["stride"]].double()
                    for t in range(0, n, 4096):
                        m = torch.zeros((min(4096, n - t), 2 * G * D), dtype=torch.float64, device="cuda")
                        for j in range(c["c"]):
                            on = live[b, l, t:t + 4096, j]
                            m += a[idx[b, l, t:t + 4096, j].clamp(min=0)] * on[:, None]
                        cnt = live[b, l, t:t + 4096].sum(-1, keepdim=True)
                        res[b, l, t:t + 4096] = (z[b, l, t:t + 4096].double() - m / cnt).float()
            return {"residual": res, "status": None}
        dist = torch.full((B, L, n, c["c"]), math.inf, dtype=torch.float64, device="cuda")
        for b in range(B):
            for l in range(L):
                a = z[b, l, ::c["stride"]].double()
                na = (a * a).sum(-1)
                for t in range(0, n, 4096):
                    x = z[b, l, t:t + 4096].double()
                    d = (x * x).sum(-1)[:, None] + na[None] - 2 * torch.matmul(x, a.T)
                    top = torch.topk(d, min(c["c"], a.shape[0]), dim=-1, largest=False, sorted=True)[0]
                    dist[b, l, t:t + 4096, :top.shape[1]] = top.clamp(min=0)
        return {"idx": None, "dist": dist, "status": None}

    H = G * c["group"]
    tk, tv = _tail(c, seed) if c["tail"] else (None, None)
    q = _queries(c, seed, max(1, c["n_q"]), 4)
    out = torch.empty(q.shape, dtype=torch.float64, device="cuda")
    sal_in = None if c["op"] == "prefill" else _salience(c, seed)
    sal_out = torch.empty((B, L, n - w), dtype=torch.float64, device="cuda")
    coef = None
    if c["op"] == "pack":
        coef = torch.zeros((B, L, G, 2, V.varrate_packed_cap_elems(_cfg(c))), dtype=torch.float64, device="cuda")
    qw = _queries(c, seed, w, 7) if c["op"] == "prefill" else None
    upto = torch.arange(n, device="cuda")[None, :] <= (n - w + torch.arange(w, device="cuda"))[:, None]
    for b in range(B):
        for l in range(L):
            if qw is not None:
                s = torch.zeros(n, dtype=torch.float64, device="cuda")
                for h in range(H):
                    x = torch.matmul(qw[l, b, :, h].double(), k[b, l, h // c["group"]].double().T) / math.sqrt(D)
                    s += torch.softmax(x.masked_fill(~upto, -math.inf), -1).sum(0)
                s = (s / (w * H))[:n - w]
                pool = 5
                sal_out[b, l] = torch.nn.functional.avg_pool1d(s[None, None], pool, 1, pool // 2, count_include_pad=True)[0, 0]
                ranks = _ranks(c, sal_out[b, l].float())
            else:
                ranks = _ranks(c, sal_in[b, l])
            keep = torch.arange(D, device="cuda")[None, :] < ranks[:, None]
            ck = torch.matmul(k[b, l].double(), bk[l].transpose(-1, -2)) * keep
            cv = torch.matmul(v[b, l].double(), bv[l].transpose(-1, -2)) * keep
            if coef is not None:
                _place(coef[b, l], ck, cv, ranks, c)
                continue
            if c["op"] == "decode_q":
                ck, cv = (_quantized(c, x.bfloat16(), ranks).double() for x in (ck, cv))
            t = (tk[l, b].double(), tv[l, b].double()) if c["tail"] else (None, None)
            out[l, b] = _attend(c, q[l, b].double(), ck, cv, ranks, bk[l], bv[l], *t)
    if c["op"] == "prefill":
        return {"salience": sal_out, "ranks": None, "attention": out, "status": None}
    if c["op"] == "pack":
        return {"ranks": None, "realized": None, "bucket_count": None, "bucket_base": None, "perm": None,
                "pos": None, "coef": coef, "status": None}
    return {"attention": out, "status": None}


def _place(coef, ck, cv, ranks, c):
    """Coefficients of one (sequence, layer) at their places of the packed layout: buckets by rank
    from r_min on, 128-slot tiles, row j's 8-slot groups turned by j."""
    base = 0
    for r in range(c["r_min"], D + 1):
        t = torch.nonzero(ranks == r).flatten()
        m = t.numel()
        n8 = -(-m // 8) * 8
        p = torch.arange(m, device=t.device)
        t0 = p // 128 * 128
        tl = torch.clamp(n8 - t0, max=128)
        j = torch.arange(r, device=t.device)
        at = base + (t0 * r)[:, None] + j[None] * tl[:, None]
        at = at + 8 * (((p - t0)[:, None] // 8 + j[None]) % (tl // 8)[:, None]) + (p % 8)[:, None]
        coef[:, 0, at] = ck[:, t, :r]
        coef[:, 1, at] = cv[:, t, :r]
        base += r * n8
