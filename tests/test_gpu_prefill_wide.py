"""Prefill scores where CTAs hold two row blocks and 256 keys: ragged tiles, odd block counts, every group
size, against float64, and an observation window of several blocks (query rows that start late)."""
import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


# 160 units and more: past one wave of 256-key CTAs and 1.5 waves of block pairs (G = 1, T <= 128: one block)
@pytest.mark.parametrize("G,D,Hkv,B,T", [
    (8, 128, 8, 20, 45), (4, 64, 8, 20, 97), (1, 64, 16, 10, 128), (1, 128, 16, 10, 129), (2, 128, 8, 20, 255),
    (2, 64, 8, 20, 257), (8, 64, 4, 20, 513), (4, 128, 8, 4, 1300)])
def test_scores_every_position(G, D, Hkv, B, T):
    torch = torch_cuda()
    g = torch.Generator(device="cuda").manual_seed(T)
    Hq, keep = G * Hkv, (T + 1) // 2 + 1               # heavy + recent > T: every position is kept
    cfg = mkv.config(mkv.MKV_H2O, B, Hq, Hkv, D, h2o_heavy=keep, h2o_recent=keep)
    cache = caches.alloc_cache(cfg, 2 * keep + 1, device="cuda")
    ws, nws = caches.workspace(cfg, max(T, 2 * keep + 1), device="cuda")
    k, v = (torch.randn((B, Hkv, T, D), generator=g, device="cuda").half() for _ in range(2))
    q = torch.randn((B, Hq, T, D), generator=g, device="cuda").half()
    mkv.mkv_h2o_prefill(cfg, q.data_ptr(), k.data_ptr(), v.data_ptr(), T, cache.c, ws.data_ptr(), nws)
    assert mkv.mkv_get_status() == 0
    late = torch.ones((T, T), dtype=torch.bool, device="cuda").triu(1)
    for b in range(B):
        s = torch.einsum("hgtd,hjd->hgtj", q[b].double().view(Hkv, G, T, D), k[b].double()) / D ** 0.5
        ref = torch.softmax(s.masked_fill(late, float("-inf")), -1).sum((1, 2))
        # fp32 products and exponents of |s| <= 40: 2^-23 * 40 of a term, twice; sums of up to 128 T / 2 terms
        # over 128 lanes and 4 warps stay below that
        torch.testing.assert_close(cache.t["acc"][b, :, :T].double(), ref, rtol=2e-5, atol=1e-6)


@pytest.mark.parametrize("G,D,B,T,W,keep", [(8, 64, 20, 600, 100, 300), (4, 128, 40, 300, 70, 111), (2, 64, 20, 1000, 200, 512)])
def test_window_of_several_blocks(G, D, B, T, W, keep):
    torch = torch_cuda()
    Hkv = 8
    cfg = mkv.config(mkv.MKV_ROCKET, B, G * Hkv, Hkv, D, snap_window=W, snap_pool=1, snap_keep=keep, topk_pages=4,
                     topq_dims=8)
    # scores that rise with a random rank, by exp(D^0.5 / 512) >= 1.5 % each: no rounding changes the order
    g = torch.Generator(device="cuda").manual_seed(T)
    rank = torch.stack([torch.randperm(T, generator=g, device="cuda") for _ in range(B * Hkv)]).view(B, Hkv, T)
    k = (rank.half() / 512)[..., None].expand(B, Hkv, T, D).contiguous()
    v = torch.randn((B, Hkv, T, D), generator=g, device="cuda").half()
    q = torch.ones((B, G * Hkv, W, D), dtype=torch.float16, device="cuda")
    c = caches.alloc_cache(cfg, (keep + 31) // 16 * 16, device="cuda")
    ws, nws = caches.workspace(cfg, T, device="cuda")
    kept = torch.full((B, Hkv, keep), -1, dtype=torch.int32, device="cuda")
    mkv.mkv_snap_compress(cfg, q.data_ptr(), k.data_ptr(), v.data_ptr(), T, c.c, kept.data_ptr(), ws.data_ptr(), nws)
    assert mkv.mkv_get_status() == 0
    best = rank[..., :T - W].topk(keep - W, -1).indices.sort(-1).values
    want = torch.cat([best, torch.arange(T - W, T, device="cuda").expand(B, Hkv, W)], -1)
    assert torch.equal(kept.long(), want)
