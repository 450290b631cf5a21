"""GPU: SnapKV's keep list where the clustered selection could go wrong -- equal scores everywhere (the
lower positions win), one planted heavy key in a long prompt (pooled scores in the workspace), prefixes
shorter than the cluster, keep one below the prompt -- and the page bounds of the gathered pages."""
import numpy as np
import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu

CASES = [  # B, Hq, Hkv, D, T, W, pool, keep, planted position
    (1, 4, 1, 64, 400001, 16, 7, 1000, 333333), (2, 8, 2, 128, 5000, 32, 7, 321, 4960), (1, 8, 8, 64, 45, 40, 3, 44, None),
    (1, 2, 1, 128, 300, 16, 1, 16, None), (3, 4, 2, 64, 1027, 16, 7, 1026, 0), (1, 8, 1, 128, 2000, 16, 5, 100, 1000),
    (1, 8, 1, 64, 900, 100, 7, 200, None), (20, 8, 8, 64, 700, 32, 7, 250, 100),
]


@pytest.mark.parametrize("B,Hq,Hkv,D,T,W,pool,keep,heavy", CASES)
def test_equal_scores_keep_lowest_positions(B, Hq, Hkv, D, T, W, pool, keep, heavy):
    torch = torch_cuda()
    dev = torch.device("cuda")
    cfg = mkv.config(mkv.MKV_ROCKET, B, Hq, Hkv, D, snap_window=W, snap_pool=pool, snap_keep=keep, topk_pages=4,
                     topq_dims=8)
    k = torch.zeros((B, Hkv, T, D), dtype=torch.float16, device=dev)
    want = list(range(keep - W))
    if heavy is not None:                      # a key every window query prefers: its neighbourhood comes first
        k[:, :, heavy] = 0.25
        near = [p for p in range(heavy - pool // 2, heavy + pool // 2 + 1) if 0 <= p < T - W]
        rest = [p for p in range(T - W) if p not in set(near)]
        want = sorted((near + rest)[:keep - W])
    v = torch.randn((B, Hkv, T, D), device=dev, generator=torch.Generator(device=dev).manual_seed(T)).half()
    q = torch.ones((B, Hq, W, D), dtype=torch.float16, device=dev)
    cap = (keep + 31) // 16 * 16
    c = caches.alloc_cache(cfg, cap, device=dev)
    ws, nws = caches.workspace(cfg, T, device=dev)
    kept = torch.full((B, Hkv, keep), -1, dtype=torch.int32, device=dev)
    for _ in range(2):                         # the workspace is left as it was found
        mkv.mkv_snap_compress(cfg, q.data_ptr(), k.data_ptr(), v.data_ptr(), T, c.c, kept.data_ptr(), ws.data_ptr(), nws)
    assert mkv.mkv_get_status() == 0
    want = torch.tensor(want + list(range(T - W, T)), dtype=torch.int32, device=dev)
    assert torch.equal(kept, want.expand(B, Hkv, keep))
    assert torch.equal(c.t["k"][:, :, :keep], k[:, :, want.long()]) and torch.equal(c.t["v"][:, :, :keep], v[:, :, want.long()])
    assert c.t["T_len"].tolist() == [keep] * B
    pg = k[:, :, want.long()][:, :, :keep // 16 * 16].unflatten(2, (keep // 16, 16))
    for name, ref in (("kmin", pg.amin(3)), ("kmax", pg.amax(3))):
        assert torch.equal(c.t[name][..., :keep // 16], ref.transpose(2, 3))
        assert not c.t[name][..., keep // 16:].any()
