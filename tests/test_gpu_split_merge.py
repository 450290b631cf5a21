"""FP16 decode at the edges of the split and of its merge: one split to hundreds, each head group size."""
import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


# (Hkv, G, D, T_cap): 1 to 3 splits, a ragged last chunk, tens of them, about 150 and about 300
@pytest.mark.parametrize("Hkv,G,D,T_cap", [
    (1, 1, 64, 64), (3, 2, 64, 65), (2, 8, 128, 130), (8, 4, 128, 4096), (1, 4, 64, 2001), (1, 2, 128, 9999),
    (2, 1, 128, 19999), (1, 8, 64, 30000), (1, 1, 128, 39000), (1, 8, 128, 39000)])
def test_split_edges(Hkv, G, D, T_cap):
    torch = torch_cuda()
    g = torch.Generator(device="cuda").manual_seed(T_cap + G)
    B, Hq = 2 if T_cap < 5000 else 1, Hkv * G
    cfg = mkv.config(mkv.MKV_FP16, B, Hq, Hkv, D)
    cache = caches.alloc_cache(cfg, T_cap, device="cuda")
    cache.t["k"].copy_(torch.randn(cache.t["k"].shape, generator=g, device="cuda"))
    cache.t["v"].copy_(torch.randn(cache.t["v"].shape, generator=g, device="cuda"))
    q = torch.randn((B, Hq, D), generator=g, device="cuda").half()
    ws, nws = caches.workspace(cfg, T_cap, device="cuda")
    for T in sorted({0, 1, T_cap // 2, T_cap - 1, T_cap}):      # the later splits hold no token
        cache.t["T_len"].fill_(T)
        out = torch.full_like(q, float("nan"))
        mkv.mkv_decode_attention(cfg, q.data_ptr(), cache.c, None, 0, out.data_ptr(), ws.data_ptr(), nws)
        k, v = (cache.t[n][:, :, :T].double().repeat_interleave(G, 1) for n in ("k", "v"))
        p = torch.softmax(torch.einsum("bhd,bhtd->bht", q.double(), k) / D ** 0.5, -1)
        ref = torch.einsum("bht,bhtd->bhd", p, v)
        # fp16 rounding of each weight (2^-11 of it) and of the result, twice over for the fp32 sums
        tol = 2.0 ** -10 * (torch.einsum("bht,bhtd->bhd", p, v.abs()) + ref.abs()) + 1e-6
        bad = (out.double() - ref).abs() > tol
        assert not bad.any() and not out.isnan().any(), (T, int(bad.sum()))
    assert mkv.mkv_get_status() == 0
