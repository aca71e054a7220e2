"""The split of the bf16 backward into local and global kernels at the sizes
where it can go wrong: no local pairs at all, no global ones, one row, tile and
step remainders on both sides of a 64- and a 128-row tile, a window edge that
falls inside a 16-key step, and groups of query heads; against the oracle's
gradients with the tolerance of the other backward tests."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("no CUDA device", allow_module_level=True)

from paper_2606_18587_gb300 import dar  # noqa: E402
from paper_2606_18587_gb300 import inputs as I  # noqa: E402
from test_gpu_backward import check, run_case  # noqa: E402


@pytest.mark.parametrize("B,Hq,Hkv,N,dd,w", [
    (1, 1, 1, 1, 16, 1),
    (1, 2, 1, 17, 16, 3),
    (2, 2, 2, 128, 16, 0),
    (1, 2, 1, 129, 32, 0),
    (1, 1, 1, 130, 64, 0),
    (1, 2, 2, 129, 16, 129),
    (1, 2, 2, 200, 32, 1000000),
    (1, 4, 2, 255, 16, 64),
    (1, 3, 1, 257, 16, 113),
    (1, 4, 1, 321, 32, 15),
    (2, 2, 1, 193, 64, 77),
], ids=lambda v: str(v))
def test_local_and_global_parts(B, Hq, Hkv, N, dd, w):
    check(run_case(I.Prefill("backward parts", 40 + N + dd, B, Hq, Hkv, N, 64, dd, w, "bf16")), "bf16")


def test_infinite_values_reach_only_the_rows_that_see_them():
    """An infinite value row changes no gradient row of a query before it, in
    whichever 16-key step or tile it lies."""
    N, w, dd = 150, 40, 16
    g = torch.Generator(device="cuda").manual_seed(1)
    q, k, v, do = (torch.empty((1, 1, N, 64), dtype=torch.bfloat16, device="cuda").normal_(generator=g)
                   for _ in range(4))
    D = torch.randn((1, 64, dd), generator=g, device="cuda") / 8
    U = torch.randn((1, dd, 64), generator=g, device="cuda") / 4
    out = dar.dar_attn_prefill(q, k, v, D, U, D, U, w)

    def grads(v):
        return dar.dar_attn_backward(q, k, v, D, U, D, U, out, do, w)["dq"]
    at = 75
    bad = v.clone()
    bad[0, 0, at, 3] = float("inf")
    a, b = grads(v), grads(bad)
    assert torch.equal(a[0, 0, :at], b[0, 0, :at])
