"""The tiled matrix-product form of the latent append: bottlenecks bit-exact
against the oracle's chain at hidden widths with and without a remainder of a
stage, widths that take the token-group kernel (not a multiple of 8), token
counts around a tile and across sequences of one tile, each tile shape, and
sequences the call refuses."""
import numpy as np
import pytest

import oracle
from paper_2606_18587_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402
from paper_2606_18587_gb300 import workloads as W  # noqa: E402


def make(B, Hkv, D, dl, w, n, before, seed):
    pages = (before + n) // 64 + 1
    table = torch.randperm(B * pages, generator=torch.Generator().manual_seed(seed)).reshape(B, pages)
    c = dar.DarLatentCache(B, Hkv, D, dl, w, pages, block_table=table)
    c.seq_lens.fill_(before)
    h = I.normal_array(seed, I.S_H, (B, n, D), dtype="bf16")
    k = I.normal_array(seed, I.S_K, (B, Hkv, n, 64), dtype="bf16")
    Wd = I.normal_array(seed, I.S_WDOWN, (D, dl), std=D ** -0.5)
    return c, table.numpy(), h, k, Wd


@pytest.mark.parametrize("B,Hkv,D,dl,w,n,before", [
    (3, 2, 64, 64, 5, 1, 0),         # 4 x 32 tiles: one token per sequence, three sequences in a tile
    (2, 1, 72, 64, 100, 17, 60),     # less than a stage; a page boundary
    (2, 2, 100, 128, 7, 33, 3),      # D not a multiple of 8: token groups
    (5, 2, 200, 192, 64, 130, 10),   # 16 x 32 tiles, a remainder of 72 past the first stage
    (2, 3, 8, 256, 16, 40, 0),       # 8 x 32 tiles, one 8-wide piece
    (4, 1, 128, 256, 50, 400, 63),   # 32 x 64 tiles, two whole stages
    (8, 2, 136, 256, 300, 450, 1),   # 32 x 64 tiles, a remainder of 8, ragged tiles
    (11, 1, 72, 256, 10, 450, 7),    # 64 x 64 tiles, a remainder of 8, a last tile of 22 rows
])
def test_bottlenecks_and_ring_are_exact(B, Hkv, D, dl, w, n, before):
    c, table, h, k, Wd = make(B, Hkv, D, dl, w, n, before, 700 + D + n)
    counts = np.array([max(1, n - 5 * b) for b in range(B)], dtype=np.int32)
    dar.dar_latent_append(c, W.upload(h, "bf16"), W.upload(k, "bf16"), W.upload(k, "bf16"), W.upload(Wd, "f32"),
                          n_per_seq=torch.from_numpy(counts).cuda())
    torch.cuda.synchronize()
    assert c.device_status() == 0
    np.testing.assert_array_equal(c.seq_lens.cpu().numpy(), before + counts)
    want = oracle.latent_bottleneck(h, Wd, "bf16")
    pool, ring, ring_v = (W.download(t) for t in (c.pool_c, c.win_k, c.win_v))
    for b in range(B):
        p = before + np.arange(counts[b])
        np.testing.assert_array_equal(pool[table[b, p // 64], p % 64], want[b, :counts[b]])
        for j in range(max(0, int(counts[b]) - w), int(counts[b])):
            np.testing.assert_array_equal(ring[b, :, (before + j) % w], k[b, :, j])
            np.testing.assert_array_equal(ring_v[b, :, (before + j) % w], k[b, :, j])


def test_refused_sequences_are_left_alone():
    c, table, h, k, Wd = make(3, 2, 64, 64, 8, 20, 0, 11)
    c.seq_lens.copy_(torch.tensor([0, 60, 5]))  # capacity 64 tokens: the second does not fit
    pool, ring = c.pool_c.clone(), c.win_k.clone()
    dar.dar_latent_append(c, W.upload(h, "bf16"), W.upload(k, "bf16"), W.upload(k, "bf16"), W.upload(Wd, "f32"),
                          n_per_seq=torch.tensor([20, 20, 21], dtype=torch.int32, device="cuda"))
    torch.cuda.synchronize()
    assert c.device_status() in (dar.DAR_ERR_INVALID_ARG, dar.DAR_ERR_CAPACITY)
    np.testing.assert_array_equal(c.seq_lens.cpu().numpy(), [20, 60, 5])
    assert torch.equal(c.win_k[1:], ring[1:]) and not torch.equal(c.win_k[0], ring[0])
    own = torch.zeros(c.num_pages, dtype=torch.bool)
    own[torch.from_numpy(table[0])] = True
    assert torch.equal(c.pool_c[~own.cuda()], pool[~own.cuda()])
