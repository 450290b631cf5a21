"""GPU: calls of different sizes from two host threads, each on its own stream: the shared-memory limit of a kernel
belongs to the function, so no call may set one that is too small for another's launch."""
import threading

import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def _caller(kind, T, torch):
    """A closure that makes one call of `kind` at size T on `stream`."""
    g = torch.Generator(device="cuda").manual_seed(T)
    B, Hq, Hkv, D, keep = 1, 2, 1, 64, 128
    cap = keep if kind == "compress" else T
    cfg = mkv.config(mkv.MKV_ROCKET, B, Hq, Hkv, D, snap_window=32, snap_pool=7, snap_keep=keep, topk_pages=4, topq_dims=16)
    c = caches.alloc_cache(cfg, cap, device="cuda")
    q = torch.randn((B, Hq, 32 if kind == "compress" else 1, D), generator=g, device="cuda").half()
    out = torch.empty((B, Hq, D), dtype=torch.float16, device="cuda")
    if kind == "compress":
        k = torch.randn((B, Hkv, T, D), generator=g, device="cuda").half()
        ws, nws = caches.workspace(cfg, T, device="cuda")
        return lambda st, keep_alive=(c, k, ws): mkv.mkv_snap_compress(cfg, q.data_ptr(), k.data_ptr(), k.data_ptr(), T, c.c, 0,
                                                                        ws.data_ptr(), nws, stream=st)
    for x in ("k", "v", "kmin", "kmax"):
        c.t[x].normal_(generator=g)
    c.t["T_len"].fill_(T)
    idx = torch.zeros((B, Hkv, 4), dtype=torch.int32, device="cuda")
    if kind == "select":
        return lambda st: mkv.mkv_rocket_select(cfg, q.data_ptr(), c.c, idx.data_ptr(), stream=st)
    return lambda st: mkv.mkv_rocket_decode(cfg, q.data_ptr(), c.c, idx.data_ptr(), out.data_ptr(), stream=st)


@pytest.mark.parametrize("kind,sizes", [("compress", (600, 100000)), ("select", (512, 100000)), ("decode", (512, 65536))])
def test_two_threads_of_different_sizes(kind, sizes):
    torch = torch_cuda()
    failed = []
    gate = threading.Barrier(2)

    def work(T):
        call, stream = _caller(kind, T, torch), torch.cuda.Stream()
        torch.cuda.synchronize()
        gate.wait()
        try:
            for i in range(3000):
                call(stream.cuda_stream)
                if i % 200 == 199:
                    stream.synchronize()
        except Exception as e:
            failed.append((T, str(e)))

    threads = [threading.Thread(target=work, args=(T,)) for T in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert not failed, failed
    assert mkv.mkv_get_status() == 0
