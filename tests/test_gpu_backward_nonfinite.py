"""Projection gradients where an infinity enters one factor: dDv = sum_j v_j^T dv^D_j with an
infinite value, dUv = sum_i O^D_i^T dO_i with an infinite dO, dDk and dUk beside them.  A
product of an infinity and a finite number is an infinity with its sign, in fp32 chains (d_down
8, fp32 storage) and on the tensor cores (bf16, from 16)."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402

INF = float("inf")


def _gradients(dtype, dd, G, spoil, N=300, w=40):
    g = torch.Generator(device="cuda").manual_seed(dd)
    B, H = 2, 2
    normal = lambda *s: torch.randn(s, device="cuda", generator=g)
    q, dout = (normal(B, H * G, N, 64).to(dtype) for _ in range(2))
    k, v = (normal(B, H, N, 64).to(dtype) for _ in range(2))
    Dk, Dv, Uk, Uv = normal(H, 64, dd) / 8, normal(H, 64, dd) / 8, normal(H, dd, 64) / 4, normal(H, dd, 64) / 4
    clean = dar.dar_attn_prefill(q, k, v, Dk, Uk, Dv, Uv, w)
    spoil(v, dout)
    # (the output of the finite inputs: what is tested is the projections' sums)
    return v, dout, dar.dar_attn_backward(q, k, v, Dk, Uk, Dv, Uv, clean, dout, w)


@pytest.mark.parametrize("G", [1, 3])
@pytest.mark.parametrize("dtype,dd", [(torch.bfloat16, 8), (torch.bfloat16, 16), (torch.bfloat16, 32),
                                      (torch.bfloat16, 64), (torch.float32, 16)])
def test_an_infinite_value(dtype, dd, G):
    """Value 7 of token 100 of one head is infinite: row 7 of that head's dDv is, with the signs of its dv^D (it has
    one, being visible globally), and the other rows and the other head are finite."""
    def spoil(v, dout):
        v[1, 1, 100, 7] = INF
    v, dout, grads = _gradients(dtype, dd, G, spoil)
    d = grads["dDv"]
    assert torch.isinf(d[1, 7]).all()
    other = torch.arange(64, device="cuda") != 7
    assert torch.isfinite(d[1][other]).all() and torch.isfinite(d[0]).all()


@pytest.mark.parametrize("dtype,dd", [(torch.bfloat16, 16), (torch.bfloat16, 32), (torch.bfloat16, 64),
                                      (torch.float32, 16)])
def test_an_infinite_output_gradient(dtype, dd):
    """dO of one row and column is infinite: that column of dUv is, and no other."""
    def spoil(v, dout):
        dout[0, 1, 200, 9] = -INF
    v, dout, grads = _gradients(dtype, dd, 1, spoil)
    d = grads["dUv"]
    assert torch.isinf(d[1, :, 9]).all()
    other = torch.arange(64, device="cuda") != 9
    assert torch.isfinite(d[1][:, other]).all() and torch.isfinite(d[0]).all()
