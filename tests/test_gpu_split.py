"""Rank allocation and layout tables over thread-block clusters: sizes at the edges of the split of a
(sequence, layer) over CTAs (one CTA up to 2048 tokens, then 2, 4 and 8; fewer with many pairs; more
tokens than shared memory holds), against the oracle bit for bit (whole numbers: no tolerance), and the
coefficients and padding that the projection writes into those tables."""
import numpy as np
import pytest
import torch

from gpu_helpers import O, V, cfg_for, coef_tol, f64, gpu_allocate, synth, unpack

pytestmark = pytest.mark.gpu


def _check(sal, wl, **kw):
    ranks, realized, status = gpu_allocate(cfg_for(wl, **kw), sal)
    flat = np.asarray(sal, np.float32).reshape(wl.batch * wl.n_layers, -1)
    for i in range(flat.shape[0]):
        want, st, tot = O.allocate_layer(flat[i], wl.n_ctx, wl.head_dim, wl.window, wl.budget_frac,
                                         wl.r_min, kw.get("mode", O.SALIENCE))
        np.testing.assert_array_equal(ranks.reshape(flat.shape[0], -1)[i], want)
        assert realized.reshape(-1)[i] == tot
    return ranks


@pytest.mark.parametrize("n_coded", [33, 1023, 2048, 2049, 4097, 8191, 8193, 16385, 32769])
@pytest.mark.parametrize("pairs", [1, 3, 40])
def test_allocation_split_edges(n_coded, pairs):
    if pairs * n_coded > 40 * 8193:
        pytest.skip("the smaller sizes cover many pairs")
    wl = synth.workload("llama1", n_ctx=n_coded + 5, window=5, n_layers=pairs, budget_frac=0.31)
    rng = np.random.default_rng(n_coded * 41 + pairs)
    _check(np.exp(1.2 * rng.standard_normal((pairs, n_coded))), wl)


@pytest.mark.parametrize("n_coded, pairs", [(1, 1), (700, 2), (2049, 1), (9000, 3), (3000, 160)])
@pytest.mark.parametrize("budget", [0.2, 0.31, 0.74])
def test_allocation_of_a_constant_salience(n_coded, pairs, budget):
    """Constant and absent (uniform mode) salience: no search, on one block and on clusters."""
    wl = synth.workload("llama1", n_ctx=n_coded + 5, window=5, n_layers=pairs, budget_frac=budget)
    for sal in (np.full((pairs, n_coded), 0.25), np.full((pairs, n_coded), np.nan)):
        got = _check(np.where(np.isnan(sal), 1.0, sal), wl)
        ranks, _, _ = gpu_allocate(cfg_for(wl), sal)
        np.testing.assert_array_equal(ranks, got)
    _check(np.random.default_rng(1).random((pairs, n_coded)), wl, mode=O.UNIFORM)


def test_allocation_more_tokens_than_shared_memory_holds():
    # 8 CTAs of 52501 tokens, of which 49152 are held normalised; one pair alone on a CTA as well
    wl = synth.workload("llama1", n_ctx=420_008, window=8, budget_frac=0.2)
    rng = np.random.default_rng(5)
    _check(np.exp(rng.standard_normal((1, 420_000))), wl)
    wl = synth.workload("llama1", n_ctx=60_008, window=8, n_layers=100, budget_frac=0.2)
    sal = np.repeat(np.exp(rng.standard_normal((1, 60_000))), 100, axis=0)
    ranks, _, _ = gpu_allocate(cfg_for(wl), sal)
    want, _, _ = O.allocate_layer(sal[0].astype(np.float32), wl.n_ctx, 128, 8, 0.2, wl.r_min, O.SALIENCE)
    np.testing.assert_array_equal(ranks.reshape(100, -1), np.broadcast_to(want, (100, wl.n_ctx)))


def test_allocation_nan_salience_is_the_floor():
    # min and max skip NaN and a NaN token keeps r_min, as a token at the minimum does
    wl = synth.workload("llama1", n_ctx=9000, window=8, budget_frac=0.3)
    rng = np.random.default_rng(6)
    sal = rng.exponential(size=(1, 8992)).astype(np.float32)
    bad = rng.random(sal.shape) < 0.05
    bad[0, np.argmin(sal)] = bad[0, np.argmax(sal)] = False
    got, _, _ = gpu_allocate(cfg_for(wl), np.where(bad, np.nan, sal))
    want, _, _ = O.allocate_layer(np.where(bad, sal.min(), sal)[0], wl.n_ctx, 128, 8, 0.3, wl.r_min, O.SALIENCE)
    np.testing.assert_array_equal(got.reshape(-1), want)


def _ranks(kind, pairs, n, r_min, rng):
    if kind == "wide":
        return rng.integers(r_min, 129, size=(pairs, n))
    if kind == "narrow":
        return np.clip(np.rint(22 + 2 * rng.standard_normal((pairs, n))), r_min, 128).astype(np.int64)
    if kind == "one":
        return np.full((pairs, n), 37)
    if kind == "mixed":   # pairs that the projection takes by token and by tile in one call
        return np.concatenate([_ranks(k, 1, n, r_min, rng) for k in ("one", "wide", "ends", "narrow")])[:pairs]
    return np.where(rng.random((pairs, n)) < 0.01, 128, r_min)   # "ends"


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("kind", ["wide", "narrow", "one", "ends"])
@pytest.mark.parametrize("n, pairs", [(9, 1), (127, 2), (129, 1), (2049, 3), (4097, 1), (8200, 1), (17001, 1),
                                      (1500, 160)])
def test_pack_split_edges(n, pairs, kind, dtype):
    _check_pack(n, pairs, kind, dtype)


@pytest.mark.parametrize("n", [700, 5003, 8200])
def test_pack_mixed_forms(n):
    _check_pack(n, 4, "mixed", "bf16")


def _check_pack(n, pairs, kind, dtype):
    """Tables bit for bit; coefficients within their storage rounding; every element of the buckets
    written (the buffer starts as NaN) and every padding slot zero."""
    if pairs > 100 and (kind != "wide" or dtype == "f32"):
        pytest.skip("one kind covers many pairs")
    r_min = 1 if kind == "ends" else 16
    wl = synth.workload("llama1", n_ctx=n, n_layers=pairs, n_kv_heads=1, window=3, budget_frac=1.0,
                        r_min=r_min, dtype=dtype)
    rng = np.random.default_rng(n * 7 + pairs)
    ranks = _ranks(kind, pairs, n, r_min, rng)
    cfg = cfg_for(wl)
    dt = synth.torch_dtype(wl)
    gen = torch.Generator().manual_seed(n)
    k, v = (torch.randn((1, pairs, 1, n, 128), generator=gen).to(dt) for _ in range(2))
    u = torch.linalg.qr(torch.randn((2, pairs, 1, 128, 128), generator=gen))[0].to(dt).contiguous()
    packed = V.PackedCache.allocate(cfg, "cuda")
    packed.coef.fill_(float("nan"))
    packed.ranks.copy_(torch.as_tensor(ranks, dtype=torch.uint8).reshape(packed.ranks.shape))
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    V.check(V.varrate_pack(cfg, k.cuda(), v.cuda(), u[0].cuda(), u[1].cuda(), packed, status), "varrate_pack")
    torch.cuda.synchronize()
    assert int(status.item()) == V.OK
    rtol, atol = coef_tol(cfg)
    for l in range(pairs) if pairs < 10 else (0, 77, pairs - 1):
        count, base, pos, perm = O.pack_tables(ranks[l], r_min, 128)
        np.testing.assert_array_equal(packed.bucket_count[0, l].cpu().numpy(), count)
        np.testing.assert_array_equal(packed.bucket_base[0, l].cpu().numpy(), base)
        np.testing.assert_array_equal(packed.pos[0, l].cpu().numpy(), pos)
        np.testing.assert_array_equal(packed.perm[0, l].cpu().numpy(), perm)
        for kv, x in ((0, k), (1, v)):
            buf = f64(packed.coef[0, l, 0, kv])
            assert np.isfinite(buf[:base[-1]]).all() and np.isnan(buf[base[-1]:]).all()
            assert np.count_nonzero(buf[:base[-1]]) <= ranks[l].sum()
            got = unpack(packed, 0, l, 0, kv, ranks[l], count, base, pos)
            want = O.truncate(O.project(f64(x[0, l, 0]), f64(u[kv, l, 0])), ranks[l])
            assert (np.abs(got - want) - (rtol * np.abs(want) + atol)).max() <= 0
