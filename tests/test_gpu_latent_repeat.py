"""Latent decode gives the same bits on every call, in shapes whose CTAs meet many
records one after the other (few rows per record, so that warps run far apart, and
the widest ones): 200 calls each, other kernels' data in L2 between them or not."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402


@pytest.mark.parametrize("B,Hq,Hkv,dl,w,lo,hi", [
    (512, 1, 1, 64, 16, 17, 300),      # a record per tile or two
    (300, 8, 8, 128, 64, 60, 700),     # eight windows of one tile beside each sequence
    (128, 32, 8, 256, 100, 100, 900),  # two row tiles, no copying warp
    (200, 20, 2, 192, 40, 41, 600),    # two row tiles with a copying warp
])
def test_every_call_gives_the_same_bits(B, Hq, Hkv, dl, w, lo, hi):
    g = torch.Generator(device="cuda").manual_seed(40 + B + Hq)
    normal = lambda *shape: torch.randn(shape, device="cuda", generator=g)
    cache = dar.DarLatentCache(B, Hkv, 64, dl, w, -(-hi // dar.PAGE_SIZE))
    for t in (cache.pool_c, cache.win_k, cache.win_v):
        t.copy_(normal(*t.shape))
    cache.seq_lens.copy_(torch.randint(lo, hi + 1, (B,), device="cuda", generator=g))
    q = normal(B, Hq, 64).bfloat16()
    A_K, A_V = normal(Hkv, 64, dl) / 8, normal(Hkv, dl, 64) / 8
    workspace = dar.latent_decode_workspace(cache, Hq)
    run = lambda: dar.dar_latent_decode(cache, q, A_K, A_V, workspace)
    first = run()
    flush = torch.empty(64 << 20, dtype=torch.float32, device="cuda")
    bad = torch.zeros(1, dtype=torch.int64, device="cuda")
    for i in range(200):
        if i % 10 == 0:
            flush.zero_()
        bad += (run() != first).sum()
    torch.cuda.synchronize()
    assert cache.device_status() == 0
    assert torch.isfinite(first).all() and int(bad.item()) == 0
