"""Scores of some 3 million log2 units, where one fp32 rounding of s * scale * log2(e) is up
to 1/8: the softmax weight of a key is 2^(s c - m), its exponent one fused multiply-add, so a
common rounding of the row's maximum m cancels and the weights stay those of exact arithmetic.
(An exponent that is rounded before m is taken off is off by up to 2^(1/4).)  The scores are
whole numbers below 2^24, exact in fp32; the tolerance is the 2e-2 of every bf16 output, of values up to 8."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402


@pytest.mark.parametrize("dd", [16, 32, 64])
@pytest.mark.parametrize("N", [33, 200])
def test_exponent_is_rounded_once(N, dd):
    r = np.random.RandomState(N + dd)
    k = np.zeros((N, 64))
    k[:, :62] = 1024.0
    k[:, 62] = r.randint(0, 21, N)
    q = np.zeros((N, 64))
    q[:, :62] = 256.0
    q[:, 62] = 1.0
    v = r.randint(-8, 9, (N, 64)).astype(float)
    s = (q @ k.T) / 8.0
    s = np.where(np.tril(np.ones((N, N))) > 0, s - s.max(), -np.inf)
    p = np.exp(s - s.max(1, keepdims=True))
    want = (p / p.sum(1, keepdims=True)) @ v
    up = lambda x: torch.tensor(x, dtype=torch.float32, device="cuda").bfloat16()[None, None].contiguous()
    z = torch.zeros(1, 64, dd, device="cuda")
    u = torch.zeros(1, dd, 64, device="cuda")
    got = dar.dar_attn_prefill(up(q), up(k), up(v), z, u, z, u, N)[0, 0].double().cpu().numpy()
    assert np.abs(got - want).max() <= 2e-2 * 8  # |v| <= 8
