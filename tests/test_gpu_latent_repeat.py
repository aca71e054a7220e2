"""Latent decode gives the same bits on every call, in shapes whose CTAs meet many
records one after the other (few rows per record, so that warps run far apart, and
the widest ones): 200 calls each, other kernels' data in L2 between them or not."""
import pytest

from paper_2606_18587_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import workloads as W  # noqa: E402


@pytest.mark.parametrize("B,Hq,Hkv,dl,w,rng", [
    (512, 1, 1, 64, 16, (17, 300)),     # a record per tile or two
    (300, 8, 8, 128, 64, (60, 700)),    # eight windows of one tile beside each sequence
    (128, 32, 8, 256, 100, (100, 900)),  # two row tiles, no copying warp
    (200, 20, 2, 192, 40, (41, 600)),   # two row tiles with a copying warp
])
def test_every_call_gives_the_same_bits(B, Hq, Hkv, dl, w, rng):
    cfg = I.LatentDecode("latent repeat", 40 + B + Hq, B, Hq, Hkv, 64, 64, dl, w, L_range=rng, shuffle_pages=True)
    wl = W.LatentDecodeWorkload(cfg, chunk=500)
    first = wl.decode().clone()
    flush = torch.empty(64 << 20, dtype=torch.float32, device="cuda")
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    for i in range(200):
        if i % 10 == 0:
            flush.zero_()
        bad += (wl.decode() != first).sum()
    torch.cuda.synchronize()
    assert wl.cache.device_status() == 0
    assert torch.isfinite(first).all() and int(bad.item()) == 0
