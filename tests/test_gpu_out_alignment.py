"""GPU: an output at any fp16 address and a workspace at any fp32 address: the merges store and read in wider pieces only
where the pointers allow it.  The output's place changes no bit; a workspace off 16 bytes is merged in another order."""
import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import assert_close, torch_cuda

pytestmark = pytest.mark.gpu


def _cache(cfg, T_cap, n, g, torch):
    c = caches.alloc_cache(cfg, T_cap, device="cuda")
    for x in ("k", "v"):
        c.t[x].normal_(generator=g)
    c.t["T_len"].fill_(n)
    if cfg.method == mkv.MKV_H2O:
        c.t["pos"][:, :, :n] = torch.arange(n, device="cuda", dtype=torch.int32)
    if cfg.method == mkv.MKV_ROCKET:
        pg = c.t["k"].unflatten(2, (T_cap // 16, 16))
        c.t["kmin"].copy_(pg.amin(3).transpose(2, 3))
        c.t["kmax"].copy_(pg.amax(3).transpose(2, 3))
    return c


def _places(B, Hq, D, torch):
    """The same output tensor shape at four addresses, one fp16 apart, with guards before and behind."""
    n = B * Hq * D
    for off in (8, 9, 10, 11):
        buf = torch.full((n + 24,), -123.0, dtype=torch.float16, device="cuda")
        yield off, buf, buf[off:off + n].view(B, Hq, D)


@pytest.mark.parametrize("method,B,Hkv,G,D,T_cap,n", [
    ("fp16", 1, 8, 4, 128, 4096, 4090), ("fp16", 2, 1, 8, 64, 300, 299), ("fp16", 1, 2, 1, 64, 64, 9), ("fp16", 1, 1, 8, 128, 39000, 39000),
    ("h2o", 2, 2, 4, 64, 701, 700), ("pages", 2, 2, 4, 128, 2048, 2000),
    ("rocket", 1, 2, 4, 64, 2048, 2000), ("rocket", 3, 8, 2, 128, 2048, 2000), ("rocket", 16, 8, 1, 64, 1024, 900)])
def test_any_output_and_workspace_address(method, B, Hkv, G, D, T_cap, n):
    torch = torch_cuda()
    g = torch.Generator(device="cuda").manual_seed(n + D)
    Hq = Hkv * G
    if method == "fp16":
        cfg = mkv.config(mkv.MKV_FP16, B, Hq, Hkv, D)
    elif method == "h2o":
        cfg = mkv.config(mkv.MKV_H2O, B, Hq, Hkv, D, h2o_heavy=400, h2o_recent=300)
    else:
        cfg = mkv.config(mkv.MKV_ROCKET, B, Hq, Hkv, D, snap_window=1, snap_keep=T_cap, topk_pages=40, topq_dims=D // 4)
    c = _cache(cfg, T_cap, n, g, torch)
    q = torch.randn((B, Hq, D), generator=g, device="cuda").half()
    nws = mkv.mkv_workspace_size(cfg, T_cap)
    room = torch.zeros(nws + 256, dtype=torch.uint8, device="cuda")
    idx = torch.full((B, Hkv, 40), -1, dtype=torch.int32, device="cuda")
    if method == "pages":
        mkv.mkv_rocket_select(cfg, q.data_ptr(), c.c, idx.data_ptr())
    outs = {}
    for shift in (0, 4, 8):
        if method == "rocket" and shift:
            continue
        for off, buf, out in _places(B, Hq, D, torch):
            if method == "rocket":
                mkv.mkv_rocket_decode(cfg, q.data_ptr(), c.c, idx.data_ptr(), out.data_ptr())
            else:
                mkv.mkv_decode_attention(cfg, q.data_ptr(), c.c, None, idx.data_ptr() if method == "pages" else 0, out.data_ptr(),
                                         room.data_ptr() + shift, nws)
            guard = torch.cat([buf[:off], buf[off + out.numel():]])
            assert bool((guard == -123.0).all()) and not bool(out.isnan().any())
            if off == 8:
                outs[shift] = out.clone()
            assert torch.equal(out, outs[shift]), (shift, off)
        assert_close(outs[shift].float().cpu(), outs[0].float().cpu(), f"workspace off by {shift}")
        room.zero_()
    assert mkv.mkv_get_status() == 0
