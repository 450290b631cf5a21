"""GPU: a prompt quantized in one call (a warp per run of tokens) leaves the cache that the same tokens
quantized one call each leave (one CTA per unit, token after token), bit for bit: codes, value ranges,
value outliers, key-outlier entries and offsets, lengths and status flags."""
import numpy as np
import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import to_dev, torch_cuda
from test_gpu_kvquant import make_cfg

pytestmark = pytest.mark.gpu


def _tokens(B, Hkv, n, D, seed, special):
    rng = np.random.default_rng(seed)
    k = rng.standard_normal((B, Hkv, n, D)) * np.exp(rng.uniform(-2, 2, (1, Hkv, 1, D)))
    v = rng.standard_normal((B, Hkv, n, D)) * np.exp(rng.uniform(-6, 6, (B, Hkv, n, 1)))
    k, v = k.astype(np.float16), v.astype(np.float16)
    if special and n >= 8:                # constant, tied, signed-zero, tiny and non-finite rows
        v[:, :, 1], k[:, :, 1] = 0.0, 0.0
        v[:, :, 2] = np.where(np.arange(D) % 2, np.float16(-0.0), np.float16(0.0))
        v[:, :, 3], k[:, :, 3] = np.float16(1.5), np.float16(-2.0)
        v[:, :, 4] = np.where(np.arange(D) % 3, np.float16(2.0), np.float16(-2.0))
        v[:, :, 5] = np.float16(6e-8) * (np.arange(D) % 5)
        v[:, :, 6, 3], k[:, :, 6, 5] = np.inf, np.inf
        v[:, :, 6, 9], k[:, :, 6, 7] = np.nan, np.nan
        v[:, :, 7, ::2], v[:, :, 7, 1::2] = np.inf, -np.inf
    return k, v


def _params(qp, Hkv, D, bits, mode, rng, order):
    K = 1 << bits
    std = np.exp(rng.uniform(-2, 2, (Hkv, D))).astype(np.float32)
    cb = np.sort(rng.standard_normal((Hkv, D, K)), axis=-1) * std[..., None]
    vcb = np.sort(rng.uniform(0, 1, (Hkv, D, K)), axis=-1)
    if order == "equal":
        cb[..., 1], vcb[..., 1] = cb[..., 0], vcb[..., 0]
    if order == "unsorted":
        cb[:, 0], vcb[:, 3] = cb[:, 0, ::-1], vcb[:, 3, ::-1]
    lo, hi = (-1.7 * std).astype(np.float32), (1.9 * std).astype(np.float32)
    lo[:, 7], hi[:, 7] = np.inf, -np.inf               # every entry an outlier
    lo[:, 8], hi[:, 8] = -1e5, 7e4                      # thresholds beyond fp16
    dev = qp.t["t_lo"].device
    for name, x in dict(t_lo=lo, t_hi=hi, k_lo=lo * 0.9, k_scale=std / K, k_cb=cb.astype(np.float16),
                        v_cb=vcb.astype(np.float16)).items():
        qp.t[name].copy_(to_dev(x, dev))
    qp.t["k_scale"][:, 2] = 0.0


def _run(cfg, qp, k, v, T_cap, cap, bulk, dev, before=0, shift=0):
    """Quantize k, v [B][Hkv][n][D] after `before` one-token calls; bulk: the rest in one call."""
    torch = torch_cuda()
    cache = caches.alloc_cache(cfg, T_cap, device=dev, k_out_cap=cap)
    n = k.shape[2]

    def call(a, b):
        m = []
        for x in (k, v):
            y = torch.empty(x[:, :, a:b].size + shift, dtype=torch.float16, device=dev)[shift:]
            y.copy_(to_dev(np.ascontiguousarray(x[:, :, a:b]).reshape(-1), dev))
            m.append(y)
        mkv.mkv_quantize_kv(cfg, qp.c, m[0].data_ptr(), m[1].data_ptr(), b - a, cache.c)
        torch.cuda.synchronize()

    for t in range(before):
        call(t, t + 1)
    if bulk:
        call(before, n)
    else:
        for t in range(before, n):
            call(t, t + 1)
    return {name: x.cpu().numpy() for name, x in cache.t.items()}, mkv.mkv_get_status()


CASES = [  # B, Hkv, D, bits, mode, frac, n, before, order
    (2, 2, 128, 4, "nuq", 0.01, 300, 0, "sorted"), (1, 8, 128, 3, "nuq", 0.01, 517, 3, "sorted"),
    (1, 3, 128, 2, "nuq", 0.01, 129, 1, "equal"), (2, 2, 64, 4, "nuq", 0.01, 70, 5, "unsorted"),
    (1, 2, 64, 3, "nuq", 0.05, 63, 0, "sorted"), (1, 2, 64, 2, "nuq", 0.0, 8, 2, "sorted"),
    (1, 2, 128, 4, "uniform", 0.01, 65, 0, "sorted"), (1, 2, 64, 3, "uniform", 0.1, 200, 7, "sorted"),
    (1, 1, 128, 2, "uniform", 0.02, 9, 1, "sorted"), (3, 1, 128, 4, "nuq", 0.06, 40, 0, "unsorted"),
    (1, 128, 64, 4, "nuq", 0.01, 150, 0, "sorted"), (1, 256, 64, 2, "nuq", 0.01, 21, 0, "sorted"),
]


@pytest.mark.parametrize("B,Hkv,D,bits,mode,frac,n,before,order", CASES)
def test_bulk_equals_token_by_token(B, Hkv, D, bits, mode, frac, n, before, order):
    torch_cuda()
    import torch
    dev = torch.device("cuda")
    rng = np.random.default_rng(n * 7 + D + bits)
    cfg = make_cfg(B, Hkv, Hkv, D, bits, mode, frac)
    qp = caches.alloc_quant_params(cfg, 1, device=dev)
    _params(qp, Hkv, D, bits, mode, rng, order)
    k, v = _tokens(B, Hkv, n, D, n + bits, special=mkv.n_value_outliers(D, frac) <= 8)
    a, fa = _run(cfg, qp, k, v, n + 3, None, False, dev, before)
    b, fb = _run(cfg, qp, k, v, n + 3, None, True, dev, before)
    assert fa == fb
    for name in a:
        assert np.array_equal(a[name].view(np.uint8), b[name].view(np.uint8)), name


def test_bulk_edges():
    """Outlier storage too small (the same entries kept, the flag), a cache without room (nothing
    written, the flag), and rows at a 2-byte address (the token-by-token kernel)."""
    torch_cuda()
    import torch
    dev = torch.device("cuda")
    B, Hkv, D, bits, n = 2, 2, 128, 4, 100
    cfg = make_cfg(B, Hkv, Hkv, D, bits, "nuq", 0.01)
    qp = caches.alloc_quant_params(cfg, 1, device=dev)
    _params(qp, Hkv, D, bits, "nuq", np.random.default_rng(1), "sorted")
    k, v = _tokens(B, Hkv, n, D, 2, special=True)
    a, fa = _run(cfg, qp, k, v, n, 333, False, dev)
    for shift in (0, 1):
        b, fb = _run(cfg, qp, k, v, n, 333, True, dev, shift=shift)
        assert fa == fb == mkv.MKV_FLAG_K_OUTLIER_OVERFLOW
        for name in a:
            assert np.array_equal(a[name].view(np.uint8), b[name].view(np.uint8)), (name, shift)
    c, fc = _run(cfg, qp, k, v, n - 1, None, True, dev, before=10)   # 10 tokens in, 90 of 89 left
    d, _ = _run(cfg, qp, k[:, :, :10], v[:, :, :10], n - 1, None, False, dev)
    assert fc == mkv.MKV_FLAG_CACHE_FULL
    for name in c:
        assert np.array_equal(c[name].view(np.uint8), d[name].view(np.uint8)), name
