"""An infinity in a visible value row comes out as an infinity in its column, and nowhere else, however many CTAs share
the keys: the direct kernels' merge has no place for a weight of zero times it."""
import pytest
import torch

from paper_2402_02082_gb300 import binding as gb
from paper_2402_02082_gb300 import build

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gb.lib()


def _inputs(B, H, H_kv, D, n, nq, dtype, at):
    gen = torch.Generator(device="cuda").manual_seed(n + D)
    cap = n + nq
    K, V = (torch.randn((B, H_kv, cap, D), generator=gen, device="cuda", dtype=dtype) for _ in range(2))
    q = torch.randn((B, nq, H, D), generator=gen, device="cuda", dtype=dtype)
    V[0, 0, at, 3] = float("inf")
    V[B - 1, H_kv - 1, at, D - 1] = float("-inf")
    code = gb.GLIDE_BF16 if dtype == torch.bfloat16 else gb.GLIDE_F32
    size = gb.glide_attn_workspace_bytes(gb.make_desc(B, H, D, cap, code, H_kv=H_kv), nq)
    ws = torch.zeros(size, dtype=torch.uint8, device="cuda")
    return q, K, V, torch.full((B,), n, dtype=torch.int32, device="cuda"), ws


def _check(out, B, H, H_kv, D):
    want = torch.zeros(out.shape, device="cuda")
    group = H // H_kv
    want[0, :, :group, 3] = float("inf")
    want[B - 1, :, H - group:, D - 1] = float("-inf")
    assert torch.equal(torch.where(torch.isinf(out), out, torch.zeros_like(out)), want)
    assert not out.isnan().any()


# splits of 1, 2, 3, 4, 5, 6 and 8 CTAs
@pytest.mark.parametrize("B,H,D,n", [(1, 4, 128, 128), (1, 4, 64, 250), (5, 16, 64, 700), (1, 4, 128, 500),
                                     (2, 24, 128, 2048), (1, 4, 64, 700), (1, 4, 128, 1024)])
@pytest.mark.parametrize("dtype", [torch.bfloat16, torch.float32])
@pytest.mark.parametrize("last", [False, True])
def test_cross(B, H, D, n, dtype, last):
    q, K, V, kv, ws = _inputs(B, H, H, D, n, 1, dtype, n - 1 if last else 5)
    _check(gb.glide_cross_attn(q, K, V, kv, n, torch.zeros((B, 1, H, D), device="cuda"), ws), B, H, H, D)


@pytest.mark.parametrize("B,H,H_kv,D,n,nq", [(1, 4, 4, 64, 100, 1), (1, 4, 2, 128, 250, 5), (2, 4, 4, 64, 500, 9),
                                             (1, 4, 4, 64, 778, 5), (1, 32, 32, 128, 300, 6), (2, 8, 2, 64, 1500, 3)])
@pytest.mark.parametrize("last", [False, True])
def test_fp32_verification(B, H, H_kv, D, n, nq, last):
    """The infinity in the prefix: every row sees it."""
    q, K, V, kv, ws = _inputs(B, H, H_kv, D, n, nq, torch.float32, n - 1 if last else 5)
    parent = torch.tensor([[-1] + [(i - 1) // 2 for i in range(1, nq)]] * B, dtype=torch.int32, device="cuda")
    _check(gb.tree_verify_attn(q, parent, K, V, kv, n, torch.zeros((B, nq, H, D), device="cuda"), ws), B, H, H_kv, D)
