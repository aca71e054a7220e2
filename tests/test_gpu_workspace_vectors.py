"""The k^D and v^D that a forward or backward call forms in its workspace are Eq. 1's
one fp32 chain, bit for bit what dar_down_project gives (and the cache append writes),
whatever the tokens beside them hold: every width, token counts around the projection's
tiles, a few and many heads (small and big tiles), an infinity and a NaN among the keys."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402

DT = {"f32": torch.float32, "bf16": torch.bfloat16}


def _bits(t):
    return t.contiguous().view(torch.int16 if t.element_size() == 2 else torch.int32)


def _inputs(dtype, B, H, N, dd, spoil):
    g = torch.Generator(device="cuda").manual_seed(100 * N + dd)
    q, k, v = (torch.randn(B, H, N, 64, device="cuda", generator=g).to(DT[dtype]) for _ in range(3))
    Dk, Dv = (torch.randn(H, 64, dd, device="cuda", generator=g) / 8 for _ in range(2))
    Uk, Uv = (torch.randn(H, dd, 64, device="cuda", generator=g) / dd ** 0.5 for _ in range(2))
    if spoil:  # rows beside them must not change how they are summed
        k[0, 0, N // 2, 3] = float("inf")
        k[-1, -1, N // 3, 60] = float("nan")
    return q, k, v, Dk, Uk, Dv, Uv


def _check(ws, at, rows, stride, want, ones):
    """Rows of `stride` elements from byte `at`: the vectors, then zeros or a block of 16 ones."""
    got = ws[at:at + rows * stride * want.element_size()].view(want.dtype).view(rows, stride)
    dd = want.shape[-1]
    assert torch.equal(_bits(got[:, :dd]), _bits(want.reshape(rows, dd)))
    pad = torch.zeros(stride - dd, device="cuda", dtype=want.dtype)
    if ones >= 0:
        pad[ones - dd:ones - dd + 16] = 1
    assert torch.equal(got[:, dd:], pad.expand(rows, -1))
    return at + (rows * stride * want.element_size() + 255) // 256 * 256


@pytest.mark.parametrize("spoil", [False, True])
@pytest.mark.parametrize("dtype,dd", [("bf16", 8), ("bf16", 16), ("bf16", 32), ("bf16", 64), ("f32", 16)])
@pytest.mark.parametrize("B,H,N", [(1, 1, 1), (1, 2, 65), (2, 3, 257), (3, 16, 2050)])
def test_forward_vectors_are_eq1_chains(dtype, dd, B, H, N, spoil):
    q, k, v, Dk, Uk, Dv, Uv = _inputs(dtype, B, H, N, dd, spoil)
    ws = torch.full((dar.dar_prefill_workspace_bytes(DT[dtype], B, H, N, dd),), 0x5a, dtype=torch.uint8, device="cuda")
    dar.dar_attn_prefill(q, k, v, Dk, Uk, Dv, Uv, 40, workspace=ws)
    bf = dtype == "bf16"
    ks = max(dd, 16) if bf else dd
    vs = {16: 32, 32: 64, 64: 64}[ks] if bf else dd
    at = _check(ws, 0, B * H * N, ks, dar.dar_down_project(k, Dk), -1)
    _check(ws, at, B * H * N, vs, dar.dar_down_project(v, Dv), ks if vs > ks else -1)


@pytest.mark.parametrize("dd", [8, 16, 32, 64])
def test_backward_vectors_are_eq1_chains(dd):
    B, H, N = 2, 2, 130
    q, k, v, Dk, Uk, Dv, Uv = _inputs("bf16", B, H, N, dd, True)
    out = dar.dar_attn_prefill(q, k, v, Dk, Uk, Dv, Uv, 40)
    ws = torch.empty(dar.dar_attn_backward_workspace_bytes(torch.bfloat16, B, H, H, N, dd), dtype=torch.uint8,
                     device="cuda")
    dar.dar_attn_backward(q, k, v, Dk, Uk, Dv, Uv, out, torch.ones_like(out), 40, workspace=ws)
    at = _check(ws, 0, B * H * N, dd, dar.dar_down_project(k, Dk), -1)
    _check(ws, at, B * H * N, dd, dar.dar_down_project(v, Dv), -1)
