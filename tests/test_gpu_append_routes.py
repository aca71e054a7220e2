"""Appends around the rules that choose a kernel and a tile for them leave the same bytes as
appends of up to eight tokens: token counts on both sides of the change to the bulk kernel
where many sequences and heads put it later than nine, and long calls of whole and of mostly
empty big tiles."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402


def _cache(B, Hkv, dd, w, pages, dtype):
    g = torch.Generator(device="cuda").manual_seed(B + dd)
    c = dar.DarCache(B, Hkv, dd, w, pages, dtype=dtype)
    for t in (c.win_k, c.win_v):
        t.normal_(generator=g)
    c.seq_lens.copy_(torch.arange(B, device="cuda") % (2 * w))  # some inside the window, some past it
    return c


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
@pytest.mark.parametrize("B,Hkv,dd,w,n", [
    (152, 8, 32, 16, 23), (152, 8, 32, 16, 24),   # 152 sequences: bulk from 24
    (153, 8, 32, 16, 12), (153, 8, 32, 16, 13),   # two waves of them: from 13
    (128, 16, 32, 16, 32), (128, 16, 32, 16, 33),
    (260, 16, 16, 16, 12), (260, 16, 16, 16, 13),
    (40, 12, 16, 33, 300),  # big tiles would be two fifths empty
    (80, 12, 16, 33, 500),  # big tiles (bf16: 2 x 256 rows for 500; fp32: 4 x 128)
    (30, 32, 64, 20, 256),
])
def test_routes_leave_the_same_bytes(B, Hkv, dd, w, n, dtype):
    pages = (2 * w + n) // dar.PAGE_SIZE + 1
    a, b = (_cache(B, Hkv, dd, w, pages, dtype) for _ in range(2))
    g = torch.Generator(device="cuda").manual_seed(n)
    k, v = (torch.randn(B, Hkv, n, 64, device="cuda", generator=g).to(dtype) for _ in range(2))
    Dk, Dv = (torch.randn(Hkv, 64, dd, device="cuda", generator=g) / 8 for _ in range(2))
    counts = torch.randint(0, n + 1, (B,), device="cuda", generator=g, dtype=torch.int32)
    counts[::3] = n
    dar.dar_cache_append(a, k, v, Dk, Dv, n_per_seq=counts)
    for j in range(0, n, 8):
        m = min(8, n - j)
        dar.dar_cache_append(b, k[:, :, j:j + m].contiguous(), v[:, :, j:j + m].contiguous(), Dk, Dv,
                             n_per_seq=(counts - j).clamp(0, m))
    torch.cuda.synchronize()
    assert a.device_status() == 0 and b.device_status() == 0
    for name in ("win_k", "win_v", "pool_kd", "pool_vd", "seq_lens"):
        assert torch.equal(getattr(a, name), getattr(b, name)), name
