"""The fp32 forward at each number of rows per CTA (8, 16, 32), with sequence
lengths around row and key tiles, against the oracle: max-abs 1e-5, the
accuracy that fp32 storage states."""
import numpy as np
import pytest

import oracle
from paper_2606_18587_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("B,Hq,Hkv,N,dd,w", [
    (1, 2, 1, 7, 8, 3),        # 8 rows: less than a tile
    (1, 4, 4, 257, 16, 65),    # 8 rows (132 CTAs), a last tile of one row and of one key
    (1, 2, 2, 128, 64, 0),     # 8 rows, whole tiles, all pairs global
    (1, 8, 4, 321, 32, 63),    # 32 rows in one wave, a last tile of one row
    (2, 8, 2, 250, 8, 1000),   # 32 rows, all pairs local
    (2, 16, 4, 193, 16, 64),   # 16 rows (two waves), a last tile of one row and of one key
    (3, 16, 8, 255, 64, 1),    # 16 rows, only the own token local
])
def test_every_row_tile(B, Hq, Hkv, N, dd, w):
    cfg = I.Prefill("case", 900 + N + dd, B, Hq, Hkv, N, 64, dd, w, "f32")
    wl = W.PrefillWorkload(cfg)
    wl.run()
    torch.cuda.synchronize()
    x = wl.host
    want = oracle.prefill(x["q"], x["k"], x["v"], x["Dk"], x["Uk"], x["Dv"], x["Uv"], cfg.w, cfg.dtype)
    got = W.to_f64(W.download(wl.out), cfg.dtype)
    assert np.isfinite(got).all()
    assert np.abs(got - want).max() <= 1e-5
