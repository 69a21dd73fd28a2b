"""The direct fp32 kernel of tree verification and grouped-query cross-attention (clusters of 1, 2,
4 or 8 CTAs per tile of 1 to 4 query rows) at the edges of its tiles, against the oracle and the
streaming kernel, which a bound on the CTAs below the direct kernel's grid selects."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_02082_gb300 import binding as gb
from paper_2402_02082_gb300 import build, synth

from gpu_util import dev

pytestmark = pytest.mark.gpu

# Two fp32 evaluations of the same softmax average of values of order 1: a sum passes through at
# most ~130 steps (a tile's keys, a warp's tiles, the warps and the CTAs), one rounding of 2^-24
# each, and scores of order 8 are off by as many roundings of 2^-22, which the weights take over:
# either is within 130 (2^-24 + 2^-22) = 3.9e-5 of exact.
AGREE = 8e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gb.lib()


@pytest.mark.parametrize("B,H,H_kv,D,kv,n,cap", [
    (1, 1, 1, 64, [0], 1, 1),                    # the root alone: one key, a cache of one row
    (2, 2, 2, 64, [0, 11], 5, 16),               # an empty sequence; keys and tree end with the tile
    (1, 4, 4, 128, [15], 16, 31),                # tree keys across a tile's end; the cache ends there
    (2, 4, 2, 128, [1000, 77], 16, 1016),        # clusters, ragged, grouped queries
    (1, 4, 4, 64, [1024], 5, 1100),              # one tree row into a second round
    (1, 8, 2, 64, [130], 64, 194),               # 256 rows a slab: tiles of 4, the longest ancestor sets
    (3, 32, 32, 128, [300, 1, 0], 7, 307),       # more tiles than a wave holds; rows that tiles do not divide
    (2, 52, 52, 64, [513, 512], 33, 546),
    (1, 2, 1, 128, [5000], 2, 5002),             # few rows, long: clusters of 8 over many rounds
    (1, 4, 2, 64, [700], 0, 700),                # n = 0: cross-attention
    (2, 12, 4, 128, [0, 129], 0, 130),
    (8, 32, 8, 128, [260, 1, 16, 17, 0, 255, 256, 128], 0, 260),
])
def test_tree_paths_agree(B, H, H_kv, D, kv, n, cap):
    rows = max(n, 1)
    K = synth.normal_values(500 + cap, 1, (B, H_kv, cap, D), "f32")
    V = synth.normal_values(500 + cap, 2, (B, H_kv, cap, D), "f32")
    q = synth.normal_values(500 + cap, 3, (B, rows, H, D), "f32")
    for b, m in enumerate(kv):  # rows past the keys are never read
        K[b, :, m + n:] = np.nan
        V[b, :, m + n:] = np.nan
    rng = np.random.default_rng(cap)
    parent = np.stack([np.asarray([-1] + [rng.integers(max(0, i - 9), i) for i in range(1, rows)], np.int32)
                       for _ in range(B)])
    if n == 64:
        parent[0] = np.arange(-1, 63)  # a chain: every earlier node is an ancestor
    desc = gb.make_desc(B, H, D, cap, gb.GLIDE_F32, H_kv=H_kv)
    ws = torch.zeros(gb.glide_attn_workspace_bytes(desc, rows), dtype=torch.uint8, device="cuda")
    qd, Kd, Vd, kvd, pd = dev(q), dev(K), dev(V), dev(np.asarray(kv, np.int32)), dev(parent)

    def run(max_ctas):
        out = torch.full((B, rows, H, D), float("nan"), device="cuda")
        if n:
            gb.tree_verify_attn(qd, pd, Kd, Vd, kvd, max(kv), out, ws, max_ctas=max_ctas)
        else:
            gb.glide_cross_attn(qd, Kd, Vd, kvd, max(kv), out, ws, max_ctas=max_ctas)
        torch.cuda.synchronize()
        return out.cpu().numpy()

    auto, again, streaming = run(0), run(0), run(1)
    assert gb.glide_read_device_status(ws) == gb.GLIDE_OK
    assert np.isfinite(auto).all()
    assert np.array_equal(auto, again), "fixed order of sums"
    assert np.abs(auto - streaming).max() <= AGREE
    want = (oracle.tree_verify_attn(q, parent, K, V, kv) if n else oracle.cross_attn(q, K, V, kv))
    assert np.abs(auto - want).max() <= AGREE


def test_tree_non_finite():
    """A NaN in a key is in the rows that see it and no others'; keys of score -inf have weight zero."""
    B, H, D, m, n = 1, 2, 64, 200, 5
    K = synth.normal_values(41, 1, (B, H, m + n, D), "f32")
    V = synth.normal_values(41, 2, (B, H, m + n, D), "f32")
    q = synth.normal_values(41, 3, (B, n, H, D), "f32")
    parent = np.asarray([[-1, 0, 0, 1, 2]], np.int32)
    q[..., 0] = 1.0
    keep = np.r_[0:16, 80:m + n]
    want = oracle.tree_verify_attn(q, parent, K[:, :, keep], V[:, :, keep], [m - 64])
    K[0, :, 16:80, 0] = -np.inf
    K[0, :, m + 1, 5] = np.nan  # node 1: seen by itself and node 3
    desc = gb.make_desc(B, H, D, m + n, gb.GLIDE_F32)
    ws = torch.zeros(gb.glide_attn_workspace_bytes(desc, n), dtype=torch.uint8, device="cuda")
    out = torch.zeros((B, n, H, D), device="cuda")
    gb.tree_verify_attn(dev(q), dev(parent), dev(K), dev(V), dev(np.asarray([m], np.int32)), m, out, ws)
    got = out.cpu().numpy()
    for i in range(n):
        if i in (1, 3):
            assert np.isnan(got[0, i]).all()
        else:
            assert np.abs(got[0, i] - want[0, i]).max() <= AGREE
