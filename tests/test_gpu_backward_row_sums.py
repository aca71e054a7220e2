"""D = dO . o of every query row, as the bf16 backward leaves it (negated) in its workspace:
chains over 8 columns whose eight sums are added pairwise, bit for bit against the same order
in numpy.  Longer chains are off by more (4 % at random inputs)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402


@pytest.mark.parametrize("dd", [16, 32, 64])
@pytest.mark.parametrize("N", [1, 77, 1030])
def test_row_sums(N, dd):
    g = torch.Generator(device="cuda").manual_seed(N + dd)
    B, H = 2, 2
    q, k, v, dout = (torch.randn(B, H, N, 64, device="cuda", generator=g).bfloat16() for _ in range(4))
    Dk, Dv = (torch.randn(H, 64, dd, device="cuda", generator=g) / 8 for _ in range(2))
    Uk, Uv = (torch.randn(H, dd, 64, device="cuda", generator=g) / dd ** 0.5 for _ in range(2))
    out = dar.dar_attn_prefill(q, k, v, Dk, Uk, Dv, Uv, 40)
    ws = torch.empty(dar.dar_attn_backward_workspace_bytes(torch.bfloat16, B, H, H, N, dd), dtype=torch.uint8,
                     device="cuda")
    dar.dar_attn_backward(q, k, v, Dk, Uk, Dv, Uv, out, dout, 40, workspace=ws)
    rows = B * H * N
    up = lambda n: (n + 255) // 256 * 256
    at = 2 * up(rows * dd * 2) + 4 * up(rows * dd * 4)  # behind k^D, v^D and four fp32 row tensors
    got = ws[at:at + rows * 4].view(torch.float32).cpu().numpy()
    x, y = (t.reshape(rows, 8, 8).double().cpu().numpy() for t in (dout, out))
    s = np.zeros((rows, 8), dtype=np.float32)
    for e in range(8):  # the products are exact in fp32
        s = (s.astype(np.float64) + x[:, :, e] * y[:, :, e]).astype(np.float32)
    while s.shape[1] > 1:
        s = s[:, 0::2] + s[:, 1::2]
    assert np.array_equal(got, -s[:, 0])
