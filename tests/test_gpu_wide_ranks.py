"""Decode and window decode on caches whose ranks spread from r_min to head_dim: buckets that are a few
slots, exactly 32 and 33 slots (where the short-tile path of the single-query kernel ends), exactly one
tile, and full tiles at every rank class of the window kernel's ring (rows rounded to 16: at most 32, 64,
128). Bars: the decode bars of gpu_helpers per output row, against the oracle on the same coefficients."""
import numpy as np
import pytest
import torch

from gpu_helpers import O, V, cfg_for, decode_close, decode_errors, f64, gpu_decode, gpu_pack, synth, unpack

pytestmark = pytest.mark.gpu


def _ranks(kind, n, rng):
    if kind == "wide":
        r = np.clip(np.rint(16 + rng.exponential(14, size=n)), 16, 128).astype(np.int64)
    elif kind == "edges":   # bucket sizes 1, 8, 9, 31, 32, 33, 127, 128, 129 at ranks of every class
        r = np.full(n, 17)
        at = 0
        for rank, m in zip((128, 127, 100, 65, 64, 63, 48, 33, 32, 31, 16), (33, 1, 8, 9, 31, 32, 33, 127, 128, 129, 40)):
            r[at:at + m] = rank
            at += m
        rng.shuffle(r)
    else:                   # full tiles of rank 128 and of r_min
        r = np.where(rng.random(n) < 0.5, 128, 16)
    return r


def _cache(kind, n, grp, dtype="bf16", G=2):
    wl = synth.workload("llama1", n_ctx=n, n_kv_heads=G, group=grp, window=3, budget_frac=1.0, r_min=16, dtype=dtype)
    rng = np.random.default_rng(n + grp)
    ranks = _ranks(kind, n, rng)
    k, v, _, bk, bv = synth.stack_inputs(wl)
    packed, st = gpu_pack(cfg_for(wl), ranks, k, v, bk, bv)
    assert st == V.OK
    ck, cv = (np.stack([O.truncate(O.project(f64(x[0, 0, g]), f64(u[0, g])), ranks) for g in range(G)])
              for x, u in ((k, bk), (v, bv)))
    return wl, cfg_for(wl), packed, bk, bv, ck, cv, ranks


@pytest.mark.parametrize("dtype, grp, n_tail", [("bf16", 4, 0), ("bf16", 7, 5), ("bf16", 1, 300), ("f32", 3, 2), ("f32", 8, 0)])
@pytest.mark.parametrize("kind, n", [("wide", 2500), ("edges", 1500), ("ends", 900)])
def test_decode_wide_ranks(kind, n, dtype, grp, n_tail):
    wl, cfg, packed, bk, bv, ck, cv, ranks = _cache(kind, n, grp, dtype)
    q = synth.stack_decode_queries(wl, 0, 1)[0]
    gen = torch.Generator().manual_seed(n_tail)
    tk, tv = (torch.randn((1, 2, n_tail, 128), generator=gen).to(synth.torch_dtype(wl)) for _ in range(2))
    tail = (tk, tv) if n_tail else (None, None)
    out, st = gpu_decode(cfg, packed, bk, bv, q, 0, *tail)
    assert st == V.OK
    want = O.decode_coef(f64(q[0]), ck, cv, ranks, f64(bk[0]), f64(bv[0]), *(f64(t[0]) for t in tail if t is not None))
    assert decode_close(out[0], want, cfg), decode_errors(out[0], want)


# rows per KV head: 32 (the mma.sync kernel), 36, 64, 65, 120, 126 and 128 (tcgen05 kernel); tails past one
# 128-token step of the combine
@pytest.mark.parametrize("grp, n_q, n_tail", [(4, 8, 150), (4, 9, 9), (8, 8, 129), (5, 13, 128), (8, 15, 257), (7, 18, 40), (4, 32, 32)])
@pytest.mark.parametrize("kind, n", [("wide", 9000), ("edges", 1500), ("ends", 4000)])
def test_window_wide_ranks(kind, n, grp, n_q, n_tail):
    wl, cfg, packed, bk, bv, ck, cv, ranks = _cache(kind, n, grp)
    q = synth.stack_decode_queries(wl, 0, n_q).permute(1, 0, 2, 3).contiguous()
    gen = torch.Generator().manual_seed(n_tail)
    tk, tv = (torch.randn((1, 2, n_tail, 128), generator=gen).to(torch.bfloat16) for _ in range(2))
    out = torch.empty_like(q, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    V.check(V.varrate_decode_window(cfg, packed, bk.cuda(), bv.cuda(), q.cuda(), n_q, 0, tk.cuda(), tv.cuda(), n_tail, out,
                                    status, V.workspace(cfg, V.CALL_DECODE_WINDOW)), "varrate_decode_window")
    torch.cuda.synchronize()
    assert int(status.item()) == V.OK
    want = O.decode_window(f64(q[0]), ck, cv, ranks, f64(bk[0]), f64(bv[0]), f64(tk[0]), f64(tv[0]))
    got = f64(out)[0]
    for i in range(n_q):
        assert decode_close(got[i], want[i], cfg), (i, decode_errors(got[i], want[i]))


@pytest.mark.parametrize("bits, grp, n_tail", [(4, 4, 0), (8, 4, 3), (4, 7, 40), (8, 1, 0)])
@pytest.mark.parametrize("kind, n", [("wide", 2500), ("edges", 1500), ("ends", 900)])
def test_decode_quantized_wide_ranks(kind, n, bits, grp, n_tail):
    """The stored bf16 coefficients are read back, so that both sides quantize the same values."""
    wl, cfg, packed, bk, bv, _, _, ranks = _cache(kind, n, grp)
    count, base, pos, _ = O.pack_tables(ranks, 16, 128)
    stored = [[unpack(packed, 0, 0, g, kv, ranks, count, base, pos) for g in range(2)] for kv in range(2)]
    ck, cv = (np.stack([O.quantize_coefficients(x.astype(np.float32), ranks, count, pos, bits)[3] for x in side])
              for side in stored)
    qp = V.QPackedCache.allocate(cfg, packed, bits)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    V.check(V.varrate_quantize(cfg, packed, qp, status), "varrate_quantize")
    q = synth.stack_decode_queries(wl, 0, 1)[0]
    gen = torch.Generator().manual_seed(n_tail)
    tk, tv = (torch.randn((1, 2, n_tail, 128), generator=gen).to(torch.bfloat16) for _ in range(2))
    out = torch.empty_like(q, device="cuda")
    V.check(V.varrate_decode_attn_q(cfg, qp, bk.cuda(), bv.cuda(), q.cuda(), 0, tk.cuda() if n_tail else None,
                                    tv.cuda() if n_tail else None, n_tail, out, status,
                                    V.workspace(cfg, V.CALL_DECODE_Q)), "varrate_decode_attn_q")
    torch.cuda.synchronize()
    assert int(status.item()) == V.OK
    want = O.decode_coef(f64(q[0]), ck.astype(np.float64), cv.astype(np.float64), ranks, f64(bk[0]), f64(bv[0]),
                         *((f64(tk[0]), f64(tv[0])) if n_tail else ()))
    got = f64(out)[0]
    assert decode_close(got, want, cfg), decode_errors(got, want)


@pytest.mark.parametrize("bits", [0, 4, 8])
def test_decode_every_rank_a_short_tile(bits):
    """Every rank from 1 to 128 holds 8 tokens, and there are more (sequence, head) pairs than thread blocks, so that
    one block takes all 128 short tiles of a pair: the largest count that the item table holds."""
    wl = synth.workload("llama1", n_ctx=1024, n_kv_heads=8, group=2, batch=32, window=3, budget_frac=1.0, r_min=1)
    cfg = cfg_for(wl)
    ranks = 1 + np.random.default_rng(0).permutation(1024) % 128
    gen = torch.Generator().manual_seed(0)
    k, v = (torch.randn((32, 1, 8, 1024, 128), generator=gen).to(torch.bfloat16) for _ in range(2))
    u = torch.linalg.qr(torch.randn((2, 1, 8, 128, 128), generator=gen))[0].to(torch.bfloat16).contiguous()
    packed, st = gpu_pack(cfg, np.tile(ranks, (32, 1, 1)), k, v, u[0], u[1])
    assert st == V.OK
    q = torch.randn((32, 16, 128), generator=gen).to(torch.bfloat16)
    if bits:
        count, base, pos, _ = O.pack_tables(ranks, 1, 128)
        qp = V.QPackedCache.allocate(cfg, packed, bits)
        status = torch.zeros(1, dtype=torch.int32, device="cuda")
        V.check(V.varrate_quantize(cfg, packed, qp, status), "varrate_quantize")
        dev = torch.empty_like(q, device="cuda")
        V.check(V.varrate_decode_attn_q(cfg, qp, u[0].cuda(), u[1].cuda(), q.cuda(), 0, None, None, 0, dev, status,
                                        V.workspace(cfg, V.CALL_DECODE_Q)), "varrate_decode_attn_q")
        assert int(status.item()) == V.OK
        out = f64(dev)
    else:
        out, st = gpu_decode(cfg, packed, u[0], u[1], q, 0)
        assert st == V.OK
    for b in (0, 13, 31):
        if bits:
            ck, cv = (np.stack([O.quantize_coefficients(unpack(packed, b, 0, g, kv, ranks, count, base, pos).astype(np.float32),
                                                        ranks, count, pos, bits)[3] for g in range(8)]).astype(np.float64)
                      for kv in range(2))
        else:
            ck, cv = (np.stack([O.truncate(O.project(f64(x[b, 0, g]), f64(w[0, g])), ranks) for g in range(8)])
                      for x, w in ((k, u[0]), (v, u[1])))
        want = O.decode_coef(f64(q[b]), ck, cv, ranks, f64(u[0][0]), f64(u[1][0]))
        assert decode_close(out[b], want, cfg), (b, decode_errors(out[b], want))
