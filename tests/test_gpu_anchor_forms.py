"""Anchor search on CTA pairs and the forms of the residual kernel, at the sizes where they change.

Search: token counts below, at and just past one CTA's 128 tokens and a pair's 256, tied distances (every
anchor twice). The distances are fp32 sums of exact products: |got - exact| <= 2^-19 (|z_t|^2 + |z_a|^2) (D =
256 terms of 2^-24 relative rounding each, and three more operations, worst case 259 * 2^-24 < 2^-15.9 of the
magnitudes' sum; random signs leave about its square root, 16 * 2^-24 = 2^-20). Residual: every operation is an
explicitly rounded fp32 one, so the result equals the same steps in torch bit for bit."""
import numpy as np
import pytest
import torch

from gpu_helpers import V

pytestmark = pytest.mark.gpu


def _kv(n, G, seed, bl=1):
    gen = torch.Generator().manual_seed(seed)
    return [torch.randn((1, bl, G, n, 128), generator=gen).to(torch.bfloat16) for _ in range(2)]


def _joint(k, v):
    return torch.cat([k, v], 2).permute(0, 1, 3, 2, 4).reshape(k.shape[1], k.shape[3], -1)


@pytest.mark.parametrize("tied", [False, True])
@pytest.mark.parametrize("n, stride, c", [(40, 8, 5), (127, 5, 4), (128, 1, 8), (129, 3, 4), (256, 16, 1), (257, 16, 8),
                                          (385, 1, 3), (1030, 2, 8)])
def test_search_pair_edges(n, stride, c, tied):
    k, v = _kv(n, 1, n + stride, bl=2)
    n_a = -(-n // stride)
    if tied:   # anchor 2 i + 1 equals anchor 2 i: the lower number comes first
        odd = torch.arange(1, n_a, 2)
        for x in (k, v):
            x[:, :, :, odd * stride] = x[:, :, :, (odd - 1) * stride]
    cfg = V.make_config(2, 1, 4, n, window=8, dtype=V.BF16)
    idx = torch.full((1, 2, n, c), -7, dtype=torch.int32, device="cuda")
    dist = torch.full((1, 2, n, c), float("nan"), device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    ws = torch.zeros(V.varrate_anchor_search_ws_bytes(cfg, stride), dtype=torch.uint8, device="cuda")
    V.check(V.varrate_anchor_search(cfg, k.cuda(), v.cuda(), stride, c, idx, dist, status, ws), "varrate_anchor_search")
    torch.cuda.synchronize()
    assert int(status.item()) == V.OK
    z = _joint(k, v).double()
    m = min(c, n_a)
    for l in range(2):
        a = z[l, ::stride]
        d = torch.cdist(z[l], a, compute_mode="donot_use_mm_for_euclid_dist") ** 2
        gi, gd = idx[0, l].cpu().long(), dist[0, l].cpu().double()
        assert (gi[:, m:] == -1).all() and torch.isinf(gd[:, m:]).all()
        gi, gd = gi[:, :m], gd[:, :m]
        assert ((gi >= 0) & (gi < n_a)).all()
        tol = 2.0 ** -19 * ((z[l] ** 2).sum(-1)[:, None] + (a ** 2).sum(-1)[gi])
        assert ((gd - d.gather(1, gi)).abs() <= tol).all()
        best = torch.topk(d, m, dim=1, largest=False)[0]
        assert ((d.gather(1, gi) - best).abs() <= 2 * tol).all()
        if m > 1:   # ordered by (reported distance, anchor)
            up, same = gd[:, 1:] > gd[:, :-1], gd[:, 1:] == gd[:, :-1]
            assert (up | (same & (gi[:, 1:] > gi[:, :-1]))).all()


@pytest.mark.parametrize("c", [1, 3, 4, 8])
@pytest.mark.parametrize("n, stride", [(700, 3), (830, 1), (831, 1), (1663, 1), (3327, 1), (6655, 1), (6656, 1)])
def test_residual_forms(n, stride, c):
    _check_residual(n, stride, c, [])


# 831 and 832 anchors: 128 and 64 columns; 1663 and 1664: 64 and 32; 3327 and 3328: 32 columns and the direct form. With
# 12287 tokens of two heads the slabs are not worth their set-up, with 12288 they are.
@pytest.mark.parametrize("c", range(1, 9))
@pytest.mark.parametrize("n, stride", [(12465, 15), (12466, 15), (13304, 8), (13305, 8), (13308, 4), (13309, 4),
                                       (12287, 16), (12288, 16)])
def test_residual_slab_forms(n, stride, c):
    _check_residual(n, stride, c, [0, 5000, n - 1])


def _check_residual(n, stride, c, bad):
    """`bad`: tokens whose lists are out of range (every other one by its last entry, the rest empty)."""
    k, v = _kv(n, 2, n + c)
    n_a = -(-n // stride)
    gen = torch.Generator().manual_seed(c)
    idx = torch.randint(0, n_a, (1, 1, n, c), generator=gen, dtype=torch.int32)
    if c > 1:
        idx[torch.rand(idx.shape, generator=gen) < 0.15] = -1
        idx[..., 0] = torch.where((idx >= 0).any(-1), idx[..., 0], n_a - 1)
    for i, t in enumerate(bad):
        idx[0, 0, t, -1 if i % 2 == 0 else slice(None)] = n_a if i % 2 == 0 else -1
    cfg = V.make_config(1, 2, 4, n, window=8, dtype=V.BF16)
    e = torch.full((1, 1, n, 512), float("nan"), dtype=torch.bfloat16, device="cuda")
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    V.check(V.varrate_anchor_residual(cfg, k.cuda(), v.cuda(), stride, c, idx.cuda(), e, status),
            "varrate_anchor_residual")
    torch.cuda.synchronize()
    assert int(status.item()) == (V.ERR_CORRUPT if bad else V.OK)
    good = torch.ones(n, dtype=torch.bool)
    good[bad] = False
    assert torch.isnan(e[0, 0].cpu()[~good]).all()
    z = _joint(k, v)[0].float()
    a, li = z[::stride], idx[0, 0].long().where(good[:, None], 0)
    acc = torch.zeros_like(z)
    for s in range(c):
        acc += torch.where(li[:, s:s + 1] >= 0, a[li[:, s].clamp(min=0)], 0.0)
    want = (z - acc / (li >= 0).sum(-1, keepdim=True).float()).to(torch.bfloat16)
    np.testing.assert_array_equal(e[0, 0].cpu()[good].view(torch.int16).numpy(), want[good].view(torch.int16).numpy())
