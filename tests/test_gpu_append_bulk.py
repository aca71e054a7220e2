"""The bulk cache append (many tokens per sequence in one call) leaves the same
bytes as appends of a few tokens each, which the one-CTA-per-sequence kernel
takes: tile edges, calls shorter and longer than the window, a context that
ends inside the window or past it, many tiles, and refused sequences."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402

FEW = 8  # tokens one round of the small kernel takes


def filled(B, Hkv, dd, w, pages, dtype, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    table = torch.randperm(B * pages, generator=torch.Generator().manual_seed(seed)).reshape(B, pages)
    c = dar.DarCache(B, Hkv, dd, w, pages, dtype=dtype, block_table=table)
    for t in (c.win_k, c.win_v):
        t.normal_(generator=g)
    Dk, Dv = (torch.randn((Hkv, 64, dd), generator=g, device="cuda") / 8 for _ in range(2))
    return c, Dk, Dv, g


def same(a, b):
    for name in ("win_k", "win_v", "pool_kd", "pool_vd", "seq_lens", "status"):
        assert torch.equal(getattr(a, name), getattr(b, name)), name


@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32], ids=["bf16", "f32"])
@pytest.mark.parametrize("B,Hkv,dd,w,n,before", [
    (3, 2, 16, 5, 9, [0, 3, 70]),           # the shortest bulk call
    (3, 1, 8, 64, 64, [0, 64, 63]),         # one whole small tile; window = call
    (3, 2, 32, 100, 65, [0, 35, 36]),       # one row past a tile; the window fills inside the call
    (2, 2, 64, 1, 129, [0, 200]),           # window of one token
    (2, 1, 16, 300, 130, [10, 500]),        # call shorter than the window
    (40, 12, 16, 33, 300, [0, 1, 40, 500]),  # many tiles, the last ones mostly empty
    (40, 12, 64, 400, 300, [7, 399]),
])
def test_bulk_equals_few_at_a_time(dtype, B, Hkv, dd, w, n, before):
    pages = (max(before) + n) // 64 + 1
    counts = [n - (b % 3) * (n // 3) for b in range(B)]
    counts[-1] = 0
    lens = torch.tensor([before[b % len(before)] for b in range(B)], dtype=torch.int32, device="cuda")
    nb = torch.tensor(counts, dtype=torch.int32, device="cuda")
    a, Dk, Dv, g = filled(B, Hkv, dd, w, pages, dtype, n + dd)
    b, _, _, _ = filled(B, Hkv, dd, w, pages, dtype, n + dd)
    k, v = (torch.empty((B, Hkv, n, 64), dtype=dtype, device="cuda").normal_(generator=g) for _ in range(2))
    a.seq_lens.copy_(lens)
    b.seq_lens.copy_(lens)
    dar.dar_cache_append(a, k, v, Dk, Dv, n_per_seq=nb)
    for j in range(0, n, FEW):
        m = min(FEW, n - j)
        dar.dar_cache_append(b, k[:, :, j:j + m].contiguous(), v[:, :, j:j + m].contiguous(), Dk, Dv,
                             n_per_seq=(nb - j).clamp(0, m))
    torch.cuda.synchronize()
    assert a.device_status() == 0
    same(a, b)


def test_refused_sequences_are_left_alone():
    """A count outside [0, n] and a length past capacity skip their sequences; the others append."""
    w, n = 16, 40
    c, Dk, Dv, g = filled(4, 2, 16, w, 2, torch.bfloat16, 3)
    c.seq_lens.copy_(torch.tensor([5, 5, 140, 20]))  # capacity: 2 pages and the window, 144 tokens
    ring = c.win_k.clone()
    k = torch.empty((4, 2, n, 64), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
    dar.dar_cache_append(c, k, k, Dk, Dv, n_per_seq=torch.tensor([n, n + 1, n, -1], dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert c.device_status() in (dar.DAR_ERR_INVALID_ARG, dar.DAR_ERR_CAPACITY)
    np.testing.assert_array_equal(c.seq_lens.cpu().numpy(), [5 + n, 5, 140, 20])
    assert torch.equal(c.win_k[1:], ring[1:])
    assert not torch.equal(c.win_k[0], ring[0])
