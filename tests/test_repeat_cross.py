"""Repeated multi-head cross-attention calls are bit-identical at full size: the direct kernel's split and the order
of its sums depend on the shapes alone."""
import pytest
import torch

from paper_2402_02082_gb300 import binding as gb
from paper_2402_02082_gb300 import build

from test_repeat import same_every_time

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gb.lib()


@pytest.mark.parametrize("B,H,D,n", [(4, 52, 128, 16384), (1, 32, 128, 2048), (4, 40, 64, 8000)])
@pytest.mark.parametrize("ragged", [False, True])
def test_multi_head_cross_repeats(B, H, D, n, ragged):
    gen = torch.Generator(device="cuda").manual_seed(B + n)
    K, V = (torch.randn((B, H, n, D), device="cuda", dtype=torch.bfloat16, generator=gen) for _ in range(2))
    q = torch.randn((B, 1, H, D), device="cuda", dtype=torch.bfloat16, generator=gen)
    lens = [n - (n // 5) * b if ragged else n for b in range(B)]
    kv = torch.tensor(lens, dtype=torch.int32, device="cuda")
    ws = torch.zeros(gb.glide_attn_workspace_bytes(gb.make_desc(B, H, D, n, gb.GLIDE_BF16), 1), dtype=torch.uint8,
                     device="cuda")
    out = torch.empty((B, 1, H, D), device="cuda")
    same_every_time(lambda: gb.glide_cross_attn(q, K, V, kv, n, out, ws), out)
