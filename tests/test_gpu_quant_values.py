"""Quantization codes at the values where a reciprocal and a division could part: quotients on and next to
the middle between two codes, constant and empty groups, subnormal steps, every tile width; against the
oracle bit for bit (codes are whole numbers and the parameters fp16 values: no tolerance)."""
import numpy as np
import pytest
import torch

from gpu_helpers import O, V, cfg_for, synth
from test_gpu_quant import _bf16, _write_stream, read_quantized

pytestmark = pytest.mark.gpu


def _values(rng, n, d):
    """Coefficients [n][d]: each column of its own kind and scale."""
    x = rng.standard_normal((n, d)) * np.exp2(rng.integers(-30, 12, size=d))
    kind = np.arange(d) % 8
    x[:, kind == 1] = rng.integers(-40, 41, size=(n, (kind == 1).sum())) * 0.5       # middles of codes
    x[:, kind == 2] = 0.1 + 0.0 * x[:, kind == 2]                                     # constant
    x[:, kind == 3] = rng.integers(0, 511, size=(n, (kind == 3).sum())) / 2.0         # middles at 8 bits
    x[:, kind == 4] = rng.integers(0, 31, size=(n, (kind == 4).sum())) / 2.0          # middles at 4 bits
    x[:, kind == 5] *= rng.random((n, (kind == 5).sum())) < 0.1                       # mostly zero
    x[:, kind == 6] = np.where(rng.random((n, (kind == 6).sum())) < 0.05, 6e4, 1e-7)  # a wide range
    return _bf16(x + 0.0)   # no negative zero


@pytest.mark.parametrize("bits", [4, 8])
@pytest.mark.parametrize("n, wide", [(700, True), (1500, False), (131, False)])
def test_quantize_codes_at_the_middles(n, wide, bits):
    wl = synth.workload("llama1", n_ctx=n, n_kv_heads=1, window=3, budget_frac=1.0, r_min=16)
    rng = np.random.default_rng(n + bits)
    ranks = rng.integers(16, 129, size=n) if wide else rng.choice([16, 19, 33, 128], size=n)
    count, base, pos, perm = O.pack_tables(ranks, 16, 128)
    cfg = cfg_for(wl)
    packed = V.PackedCache.allocate(cfg, "cuda")
    packed.bucket_count[0, 0].copy_(torch.as_tensor(count))
    packed.bucket_base[0, 0].copy_(torch.as_tensor(base))
    coefs = []
    for kv in range(2):
        c = _values(rng, n, 128) * (np.arange(128)[None, :] < ranks[:, None])
        buf = np.zeros(packed.cap_elems)
        _write_stream(buf, c, ranks, count, base, pos)
        packed.coef[0, 0, 0, kv].copy_(torch.as_tensor(buf).to(torch.bfloat16))
        coefs.append(c)
    qp = V.QPackedCache.allocate(cfg, packed, bits)
    status = torch.zeros(1, dtype=torch.int32, device="cuda")
    V.check(V.varrate_quantize(cfg, packed, qp, status), "varrate_quantize")
    torch.cuda.synchronize()
    assert int(status.item()) == V.OK
    np.testing.assert_array_equal(qp.qbase[0, 0].cpu().numpy(), O.qpack_tables(count, 16, 128, bits))
    on = np.arange(128)[None, :] < ranks[:, None]
    for kv in range(2):
        codes, lo, st = read_quantized(qp, 0, 0, 0, kv, ranks, count, pos, bits)
        wc, wlo, wst, _ = O.quantize_coefficients(coefs[kv], ranks, count, pos, bits)
        np.testing.assert_array_equal(codes[on], np.asarray(wc)[on])
        np.testing.assert_array_equal(lo[on].view(np.uint16), np.asarray(wlo).astype(np.float16)[on].view(np.uint16))
        np.testing.assert_array_equal(st[on].view(np.uint16), np.asarray(wst).astype(np.float16)[on].view(np.uint16))
