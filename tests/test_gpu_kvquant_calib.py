"""GPU: calibration at the sizes and on the data where its sorted search could go wrong -- every count
of values per thread and its edges, fewer tokens than centroids, constant, two-valued, subnormal, huge
and duplicated channels, all entries outliers -- bit for bit against the oracle."""
import numpy as np
import pytest

import paper_2609_07966_gb300 as mkv
from oracle import kvquant
from paper_2609_07966_gb300 import caches

from gpu_util import to_dev, torch_cuda
from test_gpu_kvquant import make_cfg

pytestmark = pytest.mark.gpu


def _prompt(Hkv, N, D, seed):
    rng = np.random.default_rng(seed)
    k = rng.standard_normal((Hkv, N, D)) * np.exp(rng.uniform(-3, 3, (Hkv, 1, D)))
    v = rng.standard_normal((Hkv, N, D))
    k[:, :, 0] = 3.0                                   # constant
    k[:, :, 1] = rng.integers(0, 2, (Hkv, N)) * 2 - 1  # two values
    k[:, :, 2] = rng.integers(-3, 4, (Hkv, N)) * 6e-8  # subnormal
    k[:, :, 3] *= 20000.0 / np.abs(k[:, :, 3]).max()   # huge
    k[:, :, 4] = np.rint(k[:, :, 4]) + 0.0                   # many duplicates
    k[:, N // 2, 5] = 60000.0                          # one far value
    k[:, :, 6] = np.arange(N) * 1e-3                   # ascending
    v[:, :, 0] = -8.0                                  # the token's minimum (an outlier, or u = 0)
    v[:, :, 1] = 0.0
    v[:, :, 2] = rng.integers(0, 2, (Hkv, N))
    v[:, 0] = 1.0                                      # a constant token
    if N > 4:
        v[:, 1:4] *= 1e-6                              # subnormal tokens
        v[:, 4, :9] = np.array([0, 6e-8, 1e-7, 1e-5, 1e-4, 1e-3, 100.0, 200.0, 300.0])   # u below 2^-18
    return k.astype(np.float16), v.astype(np.float16)


@pytest.mark.parametrize("bits,D,N,frac", [(4, 64, 5, 0.01), (4, 128, 17, 0.01), (3, 64, 512, 0.02), (2, 64, 513, 0.0),
                                           (4, 64, 1024, 0.3), (3, 64, 1025, 0.01), (4, 64, 2048, 0.01),
                                           (2, 128, 2049, 0.01), (4, 64, 4095, 0.01), (4, 64, 300, 1.0)])
def test_calibration_edges(bits, D, N, frac):
    torch = torch_cuda()
    dev = torch.device("cuda")
    Hkv = 2
    k, v = _prompt(Hkv, N, D, N + bits)
    cfg = make_cfg(1, Hkv, Hkv, D, bits, "nuq", frac)
    qp = caches.alloc_quant_params(cfg, 64, device=dev)
    ws, nws = caches.workspace(cfg, N, device=dev)
    kd, vd = to_dev(k, dev), to_dev(v, dev)
    mkv.mkv_kvquant_calibrate(cfg, kd.data_ptr(), vd.data_ptr(), N, N, qp.c, ws.data_ptr(), nws)
    torch.cuda.synchronize()
    ref = [kvquant.calibrate(k[h], v[h], bits, "nuq", frac) for h in range(Hkv)]
    for name, kind in (("t_lo", np.uint32), ("t_hi", np.uint32), ("k_scale", np.uint32), ("k_cb", np.uint16),
                       ("v_cb", np.uint16)):
        got, want = qp.t[name].cpu().numpy(), np.stack([getattr(p, name) for p in ref])
        bad = np.argwhere(got.view(kind) != want.view(kind))
        assert bad.size == 0, (name, bad[:4].tolist())
