"""Decode with fewer stages than the stream kernel has warps (each stage a range
of its own) and around the change to ranges of several stages (8 warps on each
SM), against the oracle: max-abs
1e-5 for fp32 storage, 2e-2 for bf16."""
import numpy as np
import pytest

import oracle
from paper_2606_18587_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("dtype,B,Hq,Hkv,dd,w,L", [
    ("bf16", 1, 1, 1, 16, 8, 1),          # one stage
    ("bf16", 1, 8, 8, 16, 128, 101),      # four ring stages per group, no pages
    ("bf16", 2, 8, 2, 32, 40, 333),       # groups of four heads, ragged ring and page stages
    ("f32", 1, 4, 4, 8, 16, 200),         # CUDA-core stages
    ("bf16", 4, 16, 16, 16, 128, 1920),   # 4 + 14 stages in each of 64 groups: 1152
    ("bf16", 4, 16, 16, 16, 128, 2048),   # 1216, the warps of 152 SMs
    ("bf16", 4, 16, 16, 16, 128, 2049),   # 1280
])
def test_small_and_borderline_splits(dtype, B, Hq, Hkv, dd, w, L):
    cfg = I.Decode("ranges", 800 + L + dd, B, Hq, Hkv, 64, dd, w, dtype, L=L, shuffle_pages=True)
    wl = W.DecodeWorkload(cfg, keep_history=True)
    out = wl.decode()
    torch.cuda.synchronize()
    assert wl.cache.device_status() == 0
    k, v = wl.history_arrays()
    Dk, Uk, Dv, Uv = wl.proj_host
    want = oracle.decode(wl.q_host, k, v, wl.lens, Dk, Uk, Dv, Uv, w, dtype)
    err = np.abs(W.to_f64(W.download(out), dtype) - want).max()
    assert err <= (1e-5 if dtype == "f32" else 2e-2), err
