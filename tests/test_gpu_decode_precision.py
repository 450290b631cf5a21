"""GPU: FP16, H2O and page-list decodes are as exact as their fp16 output allows, however many chunks share a split (and
so a maximum): the weights enter the value product with 22 bits."""
import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("method,B,Hkv,G,D,T", [
    ("fp16", 1, 8, 4, 128, 300), ("fp16", 1, 8, 4, 128, 4096), ("fp16", 1, 2, 8, 128, 8192), ("fp16", 1, 2, 4, 64, 16384),
    ("fp16", 4, 8, 4, 128, 16384), ("fp16", 2, 8, 1, 64, 5000), ("h2o", 1, 2, 8, 128, 1600), ("h2o", 2, 8, 2, 64, 3277),
    ("pages", 2, 8, 4, 128, 8192)])
def test_error_is_the_outputs_rounding(method, B, Hkv, G, D, T):
    torch = torch_cuda()
    g = torch.Generator(device="cuda").manual_seed(T + D)
    Hq, pages = Hkv * G, 128
    cfg = {"fp16": lambda: mkv.config(mkv.MKV_FP16, B, Hq, Hkv, D),
           "h2o": lambda: mkv.config(mkv.MKV_H2O, B, Hq, Hkv, D, h2o_heavy=T // 2, h2o_recent=T - T // 2 - 1),
           "pages": lambda: mkv.config(mkv.MKV_ROCKET, B, Hq, Hkv, D, snap_window=1, snap_keep=T, topk_pages=pages, topq_dims=8)}[method]()
    c = caches.alloc_cache(cfg, T, device="cuda")
    for x in ("k", "v"):
        c.t[x].normal_(generator=g)
    c.t["T_len"].fill_(T)
    held = torch.ones(T, dtype=torch.bool, device="cuda")
    idx = 0
    if method == "h2o":
        c.t["pos"].copy_(torch.arange(T, dtype=torch.int32, device="cuda"))
    if method == "pages":
        list_ = torch.arange(0, 2 * pages, 2, dtype=torch.int32, device="cuda").expand(B, Hkv, pages).contiguous()
        idx = list_.data_ptr()
        held = (torch.arange(T // 16, device="cuda") % 2 == 0) & (torch.arange(T // 16, device="cuda") < 2 * pages)
        held[-1] = True                                # the newest page is always attended
        held = held.repeat_interleave(16)
    q = torch.randn((B, Hq, D), generator=g, device="cuda").half()
    out = torch.empty_like(q)
    ws, nws = caches.workspace(cfg, T, device="cuda")
    mkv.mkv_decode_attention(cfg, q.data_ptr(), c.c, None, idx, out.data_ptr(), ws.data_ptr(), nws)
    k, v = (c.t[n][:, :, held].double().repeat_interleave(G, 1) for n in ("k", "v"))
    p = torch.softmax(torch.einsum("bhd,bhtd->bht", q.double(), k) / D ** 0.5, -1)
    ref = torch.einsum("bht,bhtd->bhd", p, v)
    # weights of 22 bits and fp32 sums add less than 1 % (in squares, 2 % of 2^-11 / sqrt(3)) to the rounding of the
    # result itself; fp16 weights add 15 to 30 %
    floor = (ref.half().double() - ref).norm()
    assert float((out.double() - ref).norm() / floor) < 1.02
    assert mkv.mkv_get_status() == 0
