"""Latent decode with as many work items (units of four pages, windows) as the main kernel has
CTAs, one fewer, one more and twice as many, against the same sums in 64 bits (max-abs 2e-2,
bf16 storage)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402


def _ctas():
    return 2 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("Hq,Hkv,dl,long_ones", [(2, 1, 64, 0), (2, 1, 128, 40), (32, 2, 256, 20), (20, 4, 192, 7)])
@pytest.mark.parametrize("more", [-1, 0, 1, "twice"])
def test_items_around_the_number_of_ctas(Hq, Hkv, dl, long_ones, more):
    w = 24
    items = 2 * _ctas() if more == "twice" else _ctas() + more
    B = (items - 2 * long_ones) // Hkv  # the long sequences have two units each, the others none
    lens = torch.randint(1, w + 1, (B,), generator=torch.Generator().manual_seed(dl))
    lens[:long_ones] = w + 300
    g = torch.Generator(device="cuda").manual_seed(dl)
    normal = lambda *shape: torch.randn(shape, device="cuda", generator=g)
    cache = dar.DarLatentCache(B, Hkv, 64, dl, w, 6)
    for t in (cache.pool_c, cache.win_k, cache.win_v):
        t.copy_(normal(*t.shape))
    cache.seq_lens.copy_(lens)
    q, A_K, A_V = normal(B, Hq, 64).bfloat16(), normal(Hkv, 64, dl) / 8, normal(Hkv, dl, 64) / dl ** 0.5
    out = dar.dar_latent_decode(cache, q, A_K, A_V, dar.latent_decode_workspace(cache, Hq))
    torch.cuda.synchronize()
    assert cache.device_status() == 0
    c = cache.pool_c.double().view(B, -1, dl)  # pages are in order
    for b in sorted({0, 1, long_ones, B // 2, B - 2, B - 1} | set(range(min(4, long_ones)))):
        L = int(lens[b])
        far, near = max(0, L - w), min(L, w)
        slots = torch.arange(L - near, L, device="cuda") % w
        k, v = (t[b][:, slots].double().repeat_interleave(Hq // Hkv, 0) for t in (cache.win_k, cache.win_v))
        ak, av = (t.double().repeat_interleave(Hq // Hkv, 0) for t in (A_K, A_V))
        x = q[b].double()
        qt = torch.einsum("ht,htc->hc", x, ak)
        s = torch.cat((torch.einsum("ht,hjt->hj", x, k), qt @ c[b, :far].T), 1) / 8
        p = s.softmax(1)
        want = torch.einsum("hj,hjt->ht", p[:, :near], v) + torch.einsum("hc,hct->ht", p[:, near:] @ c[b, :far], av)
        assert (out[b].double() - want).abs().max().item() <= 2e-2
