"""GPU: the one-call KVQuant step with more kv-heads than a batch entry's length word can count finished
CTAs of (256): its lengths advance, and its cache and outputs are those of the heads in two halves."""
import numpy as np
import pytest

import paper_2609_07966_gb300 as mkv
from paper_2609_07966_gb300 import caches

from gpu_util import assert_close, to_dev, torch_cuda
from test_gpu_kvquant import make_cfg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Hkv", [256, 258])
def test_step_many_heads(Hkv):
    torch = torch_cuda()
    dev = torch.device("cuda")
    B, D, bits, cap, half = 2, 64, 4, 70, Hkv // 2
    rng = np.random.default_rng(Hkv)

    def setup(heads):
        cfg = make_cfg(B, heads.stop - heads.start, heads.stop - heads.start, D, bits, "nuq", 0.02)
        c, qp = caches.alloc_cache(cfg, cap, device=dev), caches.alloc_quant_params(cfg, cap, device=dev)
        for name, x in params.items():
            qp.t[name].copy_(to_dev(x[heads], dev))
        mkv.mkv_quant_prepare(cfg, qp.c)
        mkv.mkv_rope_table(D, 10000.0, qp.c.rope_len, qp.t["rope"].data_ptr())
        return cfg, c, qp, caches.workspace(cfg, cap, device=dev)

    std = np.exp(rng.uniform(-1, 1, (Hkv, D))).astype(np.float32)
    params = dict(t_lo=-2 * std, t_hi=2 * std,
                  k_cb=(np.sort(rng.standard_normal((Hkv, D, 16)), -1) * std[..., None]).astype(np.float16),
                  v_cb=np.sort(rng.uniform(0, 1, (Hkv, D, 16)), -1).astype(np.float16))
    whole, parts = setup(slice(0, Hkv)), [setup(slice(0, half)), setup(slice(half, Hkv))]
    for _ in range(cap + 1):                   # the last step finds the cache full
        k, v, q = (rng.standard_normal((B, Hkv, D)).astype(np.float16) for _ in range(3))
        outs = []
        for (cfg, c, qp, (ws, nws)), h in zip([whole] + parts, (slice(0, Hkv), slice(0, half), slice(half, Hkv))):
            kd, vd, qd = (to_dev(np.ascontiguousarray(x[:, h]), dev) for x in (k, v, q))
            out = torch.empty_like(qd)
            mkv.mkv_kvquant_step(cfg, qp.c, qd.data_ptr(), kd.data_ptr(), vd.data_ptr(), c.c, out.data_ptr(),
                                 ws.data_ptr(), nws)
            outs.append(out)
        assert_close(outs[0].float().cpu(), torch.cat(outs[1:], 1).float().cpu(), "many heads")
    assert mkv.mkv_get_status() == mkv.MKV_FLAG_CACHE_FULL
    assert whole[1].t["T_len"].tolist() == [cap] * B
    for name in ("k_codes", "v_codes", "v_params", "v_out", "k_out_off", "k_out"):
        want = torch.cat([p[1].t[name] for p in parts], 1)
        assert torch.equal(whole[1].t[name].view(torch.uint8), want.view(torch.uint8)), name
