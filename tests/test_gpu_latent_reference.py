"""The reference that the latent decode's softmax weights are taken from is set anew in
every unit of four pages.  One token per unit carries the weight here (the others' scores
lie 100 below), so each weight is exactly 1 relative to its own unit and outputs are the
exact ones rounded to bf16, but for near ties: fp32 sums of five terms are off by some 2^-21,
a 2^-12 part of a bf16 step, so under 2 % of the values differ even where terms cancel.  Taken
relative to an earlier unit's maximum the weights themselves are rounded to bf16, and 21 %
differ.  And scores that fall or rise by more than fp32 can scale at once."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402

UNIT = 4 * dar.PAGE_SIZE


def _decode(B, scores, dl):
    """scores [B][units]: of the token that counts in each unit.  Returns outputs and the exact ones, columns 1.."""
    units, w = scores.shape[1], 16
    g = torch.Generator(device="cuda").manual_seed(units)
    pages = units * UNIT // dar.PAGE_SIZE + 1
    table = torch.arange(B * pages, dtype=torch.int32).view(B, pages)
    cache = dar.DarLatentCache(B, 1, 64, dl, w, pages, B * pages, block_table=table)
    c = torch.zeros(B, pages * dar.PAGE_SIZE, dl, device="cuda")
    at = torch.arange(units) * UNIT + (torch.arange(units) * 37) % UNIT
    rows = torch.randn(B, units, dl, device="cuda", generator=g).bfloat16()
    s = torch.tensor(scores, device="cuda").bfloat16()
    rows[:, :, 0] = s
    c[:, :, 0] = float(scores.min()) - 100.0
    c[:, at] = rows.float()
    cache.pool_c.copy_(c.bfloat16().view(cache.pool_c.shape))
    cache.win_k.zero_()
    cache.win_k[..., 0] = float(scores.min()) - 100.0
    cache.win_v.zero_()
    cache.seq_lens.fill_(units * UNIT + w)
    q = torch.zeros(B, 2, 64, device="cuda", dtype=torch.bfloat16)
    q[:, :, 0] = 8.0  # times the default scale of 1/8: the score is the first column
    A_K = torch.zeros(1, 64, dl, device="cuda")
    A_V = torch.zeros(1, dl, 64, device="cuda")
    for t in range(64):
        A_K[0, t, t] = A_V[0, t, t] = 1.0
    out = dar.dar_latent_decode(cache, q, A_K, A_V, dar.latent_decode_workspace(cache, 2))
    torch.cuda.synchronize()
    assert cache.device_status() == 0
    p = s.double().softmax(1)
    want = (p[:, :, None] * rows.double()).sum(1)[:, None, 1:64].expand(-1, 2, -1)
    return out[:, :, 1:], want


@pytest.mark.parametrize("dl", [64, 256])
def test_weights_of_one_are_exact(dl):
    B, units = 304, 5
    scores = np.random.RandomState(dl).uniform(-1.5, 0.0, (B, units))
    got, want = _decode(B, scores, dl)
    assert (got != want.float().bfloat16()).double().mean().item() < 0.02


@pytest.mark.parametrize("step", [-200.0, -40.0, -25.0, 40.0, 200.0])
def test_scores_that_fall_or_rise_far(step):
    got, want = _decode(304, np.tile(step * np.arange(6.0), (304, 1)), 64)
    assert (got.double() - want).abs().max().item() <= 2e-2


@pytest.mark.parametrize("units", [1, 3, 8, 9])
def test_an_infinite_record_stays_infinite(units):
    """Two tokens whose values overflow fp32 together, in a record among others: every output is the infinity that
    its weight in A_V gives it the sign of, and the sequence without them is finite."""
    dl, w = 64, 16
    cache = dar.DarLatentCache(2, 1, 64, dl, w, 4 * units + 1)
    cache.pool_c.zero_()
    cache.pool_c[0, 3, 5] = cache.pool_c[0, 4, 5] = 3.0e38
    cache.seq_lens.fill_(units * UNIT + w)
    q = torch.zeros(2, 1, 64, device="cuda", dtype=torch.bfloat16)
    A_K = torch.zeros(1, 64, dl, device="cuda")
    sign = torch.where(torch.arange(64, device="cuda") % 3 == 0, -1.0, 1.0)
    A_V = sign.expand(1, dl, 64).contiguous()
    out = dar.dar_latent_decode(cache, q, A_K, A_V, dar.latent_decode_workspace(cache, 1))
    torch.cuda.synchronize()
    assert cache.device_status() == 0
    assert torch.equal(out[0, 0].float(), sign * float("inf"))
    assert torch.equal(out[1, 0].float(), torch.zeros(64, device="cuda"))
