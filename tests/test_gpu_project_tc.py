"""The forward's own k^D and v^D: token counts around 16 rows and around a projection
tile, every width and padding (w = 0: every pair is global, so the output is all
bottleneck), against the oracle (2e-2, bf16 storage); and an infinity in one token's
key, which must reach no earlier row."""
import numpy as np
import pytest

import oracle
from paper_2606_18587_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("B,H,N,dd", [(1, 1, 1, 8), (2, 2, 15, 16), (1, 2, 17, 32), (1, 1, 63, 64), (1, 2, 65, 8),
                                      (1, 3, 257, 64), (2, 16, 1030, 16), (3, 16, 530, 32)])
def test_all_global_rows(B, H, N, dd):
    cfg = I.Prefill("projection", 600 + N + dd, B, H, H, N, 64, dd, 0, "bf16")
    wl = W.PrefillWorkload(cfg)
    wl.run()
    torch.cuda.synchronize()
    x = wl.host
    want = oracle.prefill(x["q"], x["k"], x["v"], x["Dk"], x["Uk"], x["Dv"], x["Uv"], 0, "bf16")
    assert np.abs(W.to_f64(W.download(wl.out), "bf16") - want).max() <= 2e-2


@pytest.mark.parametrize("dd", [8, 16, 32, 64])
def test_an_infinity_stays_in_its_row(dd):
    """Token 270's key holds an infinity: rows before it mask that score.  (The vectors of the tokens beside it,
    256 to 269, are Eq. 1's chains with or without it; the last bound would allow one rounding of them to bf16.)"""
    from paper_2606_18587_gb300 import dar
    g = torch.Generator(device="cuda").manual_seed(dd)
    q, k, v = (torch.randn(1, 2, 300, 64, device="cuda", generator=g).bfloat16() for _ in range(3))
    Dk, Dv = (torch.randn(2, 64, dd, device="cuda", generator=g) / 8 for _ in range(2))
    Uk, Uv = (torch.randn(2, dd, 64, device="cuda", generator=g) / dd ** 0.5 for _ in range(2))
    base = dar.dar_attn_prefill(q, k, v, Dk, Uk, Dv, Uv, 0).clone()
    k[0, 1, 270, 5] = float("inf")
    got = dar.dar_attn_prefill(q, k, v, Dk, Uk, Dv, Uv, 0)
    assert torch.equal(got[:, 0], base[:, 0])
    assert torch.equal(got[0, 1, :256], base[0, 1, :256])
    assert (got[0, 1, 256:270].float() - base[0, 1, 256:270].float()).abs().max() <= 2e-2
