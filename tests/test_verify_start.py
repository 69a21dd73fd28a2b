"""Verification where its start and its epilogue branch: a single sequence whose length is the
caller's bound, below it (the share table is made again) or, clamped, above it; and row counts
around the ones at which the 128-row kernel's warps exchange rows before they store them."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_02082_gb300 import binding as gb
from paper_2402_02082_gb300 import build, synth

from gpu_util import assert_attn_close, dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gb.lib()


def _run(B, H, H_kv, D, kv, most, n, cap):
    K = synth.normal_values(900 + n, 1, (B, H_kv, cap, D), "bf16")
    V = synth.normal_values(900 + n, 2, (B, H_kv, cap, D), "bf16")
    q = synth.normal_values(900 + n, 3, (B, n, H, D), "bf16")
    lens = [min(k, most) for k in kv]
    for b, m in enumerate(lens):
        K[b, :, m + n:] = synth.BF16_NAN
        V[b, :, m + n:] = synth.BF16_NAN
    rng = np.random.default_rng(n)
    parent = np.stack([np.asarray([-1] + [rng.integers(max(0, i - 5), i) for i in range(1, n)], np.int32)
                       for _ in range(B)])
    desc = gb.make_desc(B, H, D, cap, gb.GLIDE_BF16, H_kv=H_kv)
    ws = torch.zeros(gb.glide_attn_workspace_bytes(desc, n), dtype=torch.uint8, device="cuda")
    out = torch.full((B, n, H, D), float("nan"), device="cuda")
    gb.tree_verify_attn(dev(q), dev(parent), dev(K), dev(V), dev(np.asarray(kv, np.int32)), most, out, ws)
    torch.cuda.synchronize()
    assert gb.glide_read_device_status(ws) == gb.GLIDE_OK
    want = oracle.tree_verify_attn(q, parent, K, V, lens)
    assert_attn_close(out.cpu().numpy(), want, [(b, h) for b in range(B) for h in range(H)], f"{H}/{H_kv} {kv} {most}")


@pytest.mark.parametrize("H,H_kv", [(4, 4), (8, 2)])
@pytest.mark.parametrize("kv,most", [(300, 300), (300, 1000), (1, 1000), (0, 700), (1000, 300)])
def test_single_sequence_and_its_bound(H, H_kv, kv, most):
    _run(1, H, H_kv, 128, [kv], most, 9, 1040)


@pytest.mark.parametrize("H,H_kv,n", [
    (24, 1, 1), (25, 1, 1), (33, 1, 1),          # one warp: stored as they are, exchanged; one row in the next
    (4, 2, 28), (4, 2, 29), (8, 2, 32),          # 56, 58 and 128 rows
    (8, 2, 33), (4, 1, 64),                      # a second row tile of 4 rows; two whole ones
])
@pytest.mark.parametrize("kv", [[40], [700, 129]])
@pytest.mark.parametrize("D", [64, 128])
def test_rows_of_the_epilogue(H, H_kv, n, kv, D):
    """Slabs in one share (whole) and in several (partials)."""
    _run(len(kv), H, H_kv, D, kv, max(kv), n, max(kv) + n)
