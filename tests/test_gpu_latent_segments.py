"""Latent decode where a CTA's run of work items holds several units of one
sequence (one record, the other slots empty), several sequences and windows, and
where one KV head has more than 16 query heads, against the oracle (max-abs
2e-2, bf16 storage with fp32 accumulation)."""
import numpy as np
import pytest

import oracle
from paper_2606_18587_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("B,Hq,Hkv,D,dl,w,rng", [
    (2, 32, 1, 64, 64, 70, (60, 400)),     # 32 query heads on one KV head, short and long of the window
    (3, 24, 1, 64, 256, 20, (100, 300)),   # 24: a partly filled second row tile
    (96, 2, 1, 64, 64, 64, (1, 2000)),     # about 340 units and 96 windows over 304 CTAs
    (200, 4, 2, 64, 192, 130, (700, 900)),  # about 600 units and 400 windows
])
def test_runs_of_items(B, Hq, Hkv, D, dl, w, rng):
    cfg = I.LatentDecode("latent runs", 900 + B + Hq, B, Hq, Hkv, 64, D, dl, w, L_range=rng, shuffle_pages=True)
    wl = W.LatentDecodeWorkload(cfg, keep_history=True, chunk=500)
    out = wl.decode()
    torch.cuda.synchronize()
    assert wl.cache.device_status() == 0
    got = W.to_f64(W.download(out), "bf16")
    assert np.isfinite(got).all()
    seqs = list(range(0, B, max(1, B // 24)))
    k, v, h = wl.history_arrays(seqs)
    Wdown, Wup, WK, WV = wl.proj_host
    heads = [(i, hq) for i in range(len(seqs)) for hq in range(Hq)]
    want = oracle.latent_decode(np.ascontiguousarray(wl.q_host[seqs]), k, v, h, wl.lens[seqs], Wdown, Wup, WK, WV,
                                w, "bf16", heads=heads)
    assert max(np.abs(got[seqs[i], hq] - want[i, hq]).max() for i, hq in heads) <= 2e-2
