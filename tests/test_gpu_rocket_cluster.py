"""GPU: the one-launch RocketKV step at every cluster size and where its page choice could go wrong
(tied and equal scores, one page to several thousand, budgets from one page to all of them) against the
two calls it stands for: mkv_rocket_select must list the same pages (integer inputs make the scores
exact in any order) and mkv_decode_attention over them agree within the attention tolerance."""
import numpy as np
import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import assert_close, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

CASES = [  # B, Hq, Hkv, D, slots held, slots, pages chosen, dims, values
    (1, 8, 8, 128, 4097, 4160, 64, 32, "ties"), (3, 32, 8, 128, 700, 720, 9, 32, "ties"),
    (9, 32, 8, 128, 1040, 1056, 20, 40, "plain"), (10, 8, 8, 64, 333, 336, 5, 16, "ties"),
    (15, 16, 8, 64, 4112, 4128, 100, 16, "ties"), (20, 32, 8, 128, 500, 512, 40, 32, "plain"),
    (1, 8, 1, 128, 16400, 16432, 257, 128, "ties"), (1, 8, 2, 64, 40000, 40016, 300, 3, "ties"),
    (2, 8, 2, 64, 777, 784, 48, 16, "equal"), (130, 1, 1, 64, 2000, 2000, 11, 16, "equal"),
    (1, 2, 2, 128, 1, 16, 4, 8, "plain"), (1, 4, 2, 64, 16, 32, 4, 8, "plain"), (2, 4, 2, 64, 17, 32, 1, 8, "plain"),
    # at most 128 candidate pages counted, up to 1023 by two bits a round, more by one
    (1, 8, 4, 64, 2064, 2080, 33, 16, "ties"), (2, 8, 8, 64, 2065, 2080, 128, 16, "ties"),
    (1, 8, 2, 64, 16384, 16400, 200, 16, "ties"), (1, 8, 2, 128, 16385, 16400, 200, 16, "plain"),
    (1, 8, 2, 64, 5000, 5008, 31, 16, "equal"), (3, 8, 2, 64, 2000, 2000, 124, 16, "equal"),
]


@pytest.mark.parametrize("B,Hq,Hkv,D,n,cap,pages,dims,values", CASES)
def test_fused_equals_two_calls(B, Hq, Hkv, D, n, cap, pages, dims, values):
    torch = torch_cuda()
    dev = torch.device("cuda")
    rng = np.random.default_rng(n + B)
    if values == "plain":
        k = rng.integers(-9, 10, (B, Hkv, cap, D)) / 8
    else:
        k = rng.integers(0 if values == "equal" else -1, 1 if values == "equal" else 2, (B, Hkv, cap, D)) * 1.0
    q = rng.integers(-3, 4, (B, Hq, D)) / 4
    cfg = mkv.config(mkv.MKV_ROCKET, B, Hq, Hkv, D, snap_window=1, snap_keep=cap, topk_pages=pages, topq_dims=dims)
    c = caches.alloc_cache(cfg, cap, device=dev)
    c.t["k"].copy_(to_dev(k.astype(np.float16), dev))
    c.t["v"].normal_(generator=torch.Generator(device=dev).manual_seed(n))
    pg = c.t["k"].unflatten(2, (cap // 16, 16))
    c.t["kmin"].copy_(pg.amin(3).transpose(2, 3))
    c.t["kmax"].copy_(pg.amax(3).transpose(2, 3))
    c.t["T_len"].fill_(n)
    if B > 2:
        c.t["T_len"][1] = 0                                 # an empty entry and a short one
        c.t["T_len"][2] = min(n, 20)
    qd = to_dev(q.astype(np.float16), dev)
    ws, nws = caches.workspace(cfg, cap, device=dev)
    idx, idx2 = (torch.full((B, Hkv, pages), -7, dtype=torch.int32, device=dev) for _ in range(2))
    out, out2 = torch.empty_like(qd), torch.empty_like(qd)
    mkv.mkv_rocket_select(cfg, qd.data_ptr(), c.c, idx.data_ptr())
    mkv.mkv_decode_attention(cfg, qd.data_ptr(), c.c, None, idx.data_ptr(), out.data_ptr(), ws.data_ptr(), nws)
    mkv.mkv_rocket_decode(cfg, qd.data_ptr(), c.c, idx2.data_ptr(), out2.data_ptr())
    assert torch.equal(idx, idx2)
    assert_close(out2.float().cpu(), out.float().cpu(), "fused against two calls")
    assert mkv.mkv_get_status() == 0


@pytest.mark.parametrize("Hkv,D,T_cap,dims", [(4, 64, 32, 32), (4, 64, 4160, 32), (2, 128, 8192, 128), (25, 64, 4160, 32),
                                              (16, 64, 4160, 64)])
def test_no_candidate_page(Hkv, D, T_cap, dims):
    """At most 16 tokens in a cache of any capacity (one head a group, so that the page bounds of the capacity are
    larger than a CTA's partial): the newest page is the whole result, in every call the same bits."""
    torch = torch_cuda()
    dev = torch.device("cuda")
    lens = [1, 2, 15, 16]
    B, reps = len(lens), 50
    g = torch.Generator(device=dev).manual_seed(T_cap + Hkv)
    cfg = mkv.config(mkv.MKV_ROCKET, B, Hkv, Hkv, D, snap_window=1, snap_keep=T_cap, topk_pages=3, topq_dims=dims)
    c = caches.alloc_cache(cfg, T_cap, device=dev)
    for name in ("k", "v", "kmin", "kmax"):            # (bounds of pages that do not exist: never looked at)
        c.t[name].normal_(generator=g)
    q = torch.randn((B, Hkv, D), device=dev, generator=g).half()
    n = torch.tensor(lens, dtype=torch.int32, device=dev)
    c.t["T_len"].copy_(n)
    k, v = (c.t[x][:, :, :16].double() for x in ("k", "v"))
    s = torch.einsum("bhd,bhtd->bht", q.double(), k) / D ** 0.5
    s = s.masked_fill(torch.arange(16, device=dev) >= n[:, None, None], float("-inf"))
    ref = torch.einsum("bht,bhtd->bhd", torch.softmax(s, -1), v)
    idx = torch.full((reps, B, Hkv, 3), -7, dtype=torch.int32, device=dev)
    out = torch.full((2 * reps, B, Hkv, D), float("nan"), dtype=torch.float16, device=dev)
    for i in range(reps):
        mkv.mkv_rocket_decode(cfg, q.data_ptr(), c.c, idx[i].data_ptr(), out[i].data_ptr())
    kn, vn = (torch.stack([c.t[x][b, :, lens[b] - 1] for b in range(B)]) for x in ("k", "v"))
    for i in range(reps):                              # the same with the last token appended by the step
        c.t["T_len"].copy_(n - 1)
        mkv.mkv_rocket_step(cfg, q.data_ptr(), kn.data_ptr(), vn.data_ptr(), c.c, 0, out[reps + i].data_ptr())
    assert mkv.mkv_get_status() == 0 and torch.equal(c.t["T_len"], n) and bool((idx == -1).all())
    assert_close(out[0].double().cpu(), ref.cpu(), "newest page alone")
    assert bool((out == out[0]).all())


# units at each preferred cluster size, with the longest cache the step accepts: where the bounds and partial scores
# of a CTA's pages do not fit, more CTAs share a unit
@pytest.mark.parametrize("B,Hkv,D,dims", [(2, 8, 128, 128), (4, 8, 128, 128), (4, 16, 128, 32), (16, 4, 128, 128), (7, 16, 128, 64),
                                          (8, 16, 128, 32), (8, 16, 128, 128), (32, 8, 128, 64), (8, 16, 64, 16), (14, 8, 64, 64)])
def test_longest_accepted_cache(B, Hkv, D, dims):
    torch = torch_cuda()
    dev = torch.device("cuda")
    T_cap, G, pages, steps = 32768 if D == 128 else 65536, 4 if D == 128 else 2, 9, 3
    g = torch.Generator(device=dev).manual_seed(B * Hkv + dims)
    cfg = mkv.config(mkv.MKV_ROCKET, B, G * Hkv, Hkv, D, snap_window=1, snap_keep=T_cap, topk_pages=pages, topq_dims=dims)
    twins = [caches.alloc_cache(cfg, T_cap, device=dev) for _ in range(2)]
    a, c = twins
    for name in ("k", "v"):                            # integers: page scores are exact in any order
        a.t[name].copy_(torch.randint(-9, 10, a.t[name].shape, generator=g, device=dev, dtype=torch.int8))
        a.t[name].div_(8)
    pg = a.t["k"].unflatten(2, (T_cap // 16, 16))
    a.t["kmin"].copy_(pg.amin(3).transpose(2, 3))
    a.t["kmax"].copy_(pg.amax(3).transpose(2, 3))
    a.t["T_len"].fill_(T_cap - 2)                      # the last step finds the cache full
    a.t["T_len"][0] = 5000
    for name in a.t:
        c.t[name].copy_(a.t[name])
    ws, nws = caches.workspace(cfg, T_cap, device=dev)
    for s in range(steps):
        q = torch.randint(-3, 4, (B, G * Hkv, D), generator=g, device=dev).half() / 4
        kn, vn = (torch.randint(-9, 10, (B, Hkv, D), generator=g, device=dev).half() / 8 for _ in range(2))
        idx, idx1 = (torch.full((B, Hkv, pages), -7, dtype=torch.int32, device=dev) for _ in range(2))
        ref, out, out1 = torch.empty_like(q), torch.empty_like(q), torch.empty_like(q)
        full = (0, mkv.MKV_FLAG_CACHE_FULL)[s == steps - 1]
        mkv.mkv_append_kv(cfg, kn.data_ptr(), vn.data_ptr(), a.c)
        assert mkv.mkv_get_status() == full
        mkv.mkv_rocket_select(cfg, q.data_ptr(), a.c, idx.data_ptr())
        mkv.mkv_decode_attention(cfg, q.data_ptr(), a.c, None, idx.data_ptr(), ref.data_ptr(), ws.data_ptr(), nws)
        mkv.mkv_rocket_decode(cfg, q.data_ptr(), a.c, idx1.data_ptr(), out1.data_ptr())
        assert torch.equal(idx, idx1)
        mkv.mkv_rocket_step(cfg, q.data_ptr(), kn.data_ptr(), vn.data_ptr(), c.c, idx1.fill_(-7).data_ptr(), out.data_ptr())
        assert mkv.mkv_get_status() == full
        assert torch.equal(idx, idx1) and torch.equal(out, out1)
        assert_close(out.float().cpu(), ref.float().cpu(), f"step {s}")
        for name in a.t:
            assert torch.equal(a.t[name], c.t[name]), (s, name)


@pytest.mark.parametrize("n,pages", [(1600, 9), (4160, 64), (16400, 200), (32000, 30)])
@pytest.mark.parametrize("D,dims", [(64, 16), (128, 32)])
def test_nan_and_infinite_values_choose_real_pages(D, dims, n, pages):
    """A query with NaNs or infinite cached keys in one batch entry: its page list still holds distinct pages in range and
    nothing is written behind it, and the other entry is not touched."""
    torch = torch_cuda()
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(n)
    B, Hkv, G = 4, 2, 4
    cap = (n + 31) // 16 * 16
    cfg = mkv.config(mkv.MKV_ROCKET, B, Hkv * G, Hkv, D, snap_window=1, snap_keep=cap, topk_pages=pages, topq_dims=dims)
    c = caches.alloc_cache(cfg, cap, device=dev)
    for x in ("k", "v"):
        c.t[x].normal_(generator=g)
    c.t["k"][1, :, ::37, ::3] = float("inf")
    c.t["k"][1, :, 5::61, 1::3] = float("-inf")
    pg = c.t["k"].unflatten(2, (cap // 16, 16))
    c.t["kmin"].copy_(pg.amin(3).transpose(2, 3))
    c.t["kmax"].copy_(pg.amax(3).transpose(2, 3))
    c.t["T_len"].fill_(n)
    clean = torch.randn((B, Hkv * G, D), generator=g, device=dev).half()
    q = clean.clone()
    q[1, :, ::2] = q[1, :, ::2].clamp(min=0)           # (0 * inf)
    q[2, 1, ::5] = float("nan")
    q[3] = float("nan")
    ns = (n - 1) // 16
    for call in ("select", "fused"):
        lists = {}
        for name, x in (("clean", clean), ("q", q)):
            buf = torch.full((B * Hkv * pages + 64,), -77, dtype=torch.int32, device=dev)
            out = torch.empty_like(q)
            if call == "select":
                mkv.mkv_rocket_select(cfg, x.data_ptr(), c.c, buf.data_ptr())
            else:
                mkv.mkv_rocket_decode(cfg, x.data_ptr(), c.c, buf.data_ptr(), out.data_ptr())
                assert not bool(out[0].isnan().any())
            assert mkv.mkv_get_status() == 0
            assert bool((buf[B * Hkv * pages:] == -77).all())
            lists[name] = buf[:B * Hkv * pages].view(B, Hkv, pages)
        x = lists["q"]
        assert torch.equal(x[0], lists["clean"][0])
        assert bool((x >= 0).all() and (x < ns).all() and (x[..., 1:] > x[..., :-1]).all())


# units whose clusters have 4, 2 and 1 CTAs
@pytest.mark.parametrize("B,Hkv,G,D", [(4, 8, 4, 128), (7, 8, 1, 64), (14, 8, 2, 64), (10, 10, 4, 128), (16, 8, 4, 128), (33, 4, 8, 64)])
def test_step_equals_append_then_decode_beyond_16_units(B, Hkv, G, D):
    """mkv_rocket_step against mkv_append_kv + mkv_rocket_decode on twin caches, bit for bit: empty and one-page entries,
    pages completed, caches that fill up."""
    torch = torch_cuda()
    dev = torch.device("cuda")
    g = torch.Generator(device=dev).manual_seed(B * D)
    T_cap, steps, pages = 112, 20, 3
    cfg = mkv.config(mkv.MKV_ROCKET, B, Hkv * G, Hkv, D, snap_window=1, snap_keep=T_cap, topk_pages=pages, topq_dims=D // 4)
    a, c = (caches.alloc_cache(cfg, T_cap, device=dev) for _ in range(2))
    for x in ("k", "v"):
        a.t[x].normal_(generator=g)
    pg = a.t["k"].unflatten(2, (T_cap // 16, 16))
    a.t["kmin"].copy_(pg.amin(3).transpose(2, 3))
    a.t["kmax"].copy_(pg.amax(3).transpose(2, 3))
    a.t["T_len"].copy_(torch.tensor([[0, 15, 16, 47, 60, 100, 112][b % 7] for b in range(B)], dtype=torch.int32))
    for x in a.t:
        c.t[x].copy_(a.t[x])
    for s in range(steps):
        q = torch.randn((B, Hkv * G, D), generator=g, device=dev).half()
        kn, vn = (torch.randn((B, Hkv, D), generator=g, device=dev).half() for _ in range(2))
        ia, ic = (torch.full((B, Hkv, pages), -7, dtype=torch.int32, device=dev) for _ in range(2))
        oa, oc = torch.empty_like(q), torch.empty_like(q)
        mkv.mkv_append_kv(cfg, kn.data_ptr(), vn.data_ptr(), a.c)
        fa = mkv.mkv_get_status()
        mkv.mkv_rocket_decode(cfg, q.data_ptr(), a.c, ia.data_ptr(), oa.data_ptr())
        mkv.mkv_rocket_step(cfg, q.data_ptr(), kn.data_ptr(), vn.data_ptr(), c.c, ic.data_ptr(), oc.data_ptr())
        assert mkv.mkv_get_status() == fa
        assert torch.equal(oa, oc) and torch.equal(ia, ic), s
        for x in a.t:
            assert torch.equal(a.t[x], c.t[x]), (s, x)
    assert fa == mkv.MKV_FLAG_CACHE_FULL if B >= 6 else fa == 0
