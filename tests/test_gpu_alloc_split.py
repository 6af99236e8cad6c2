"""Rank allocation over thread-block clusters: sizes at the edges of the split of a (sequence, layer)
over CTAs (one CTA up to 2048 tokens, then 2, 4 and 8; fewer with many pairs; more tokens than shared
memory holds), against the oracle bit for bit. Ranks are whole numbers: no tolerance."""
import numpy as np
import pytest

from gpu_helpers import O, V, cfg_for, gpu_allocate, synth

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
