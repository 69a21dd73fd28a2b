"""Which kernel serves multi-head cross-attention, and that both agree: the
direct kernel (clusters of 1, 2, 4 or 8 CTAs per (sequence, head), one or
several waves of them) at the edges of its tiles and rounds, and the streaming
kernel, which a bound on the CTAs below the direct kernel's grid selects, and
which serves few heads over more than 8192 keys."""
import numpy as np
import pytest
import torch

import oracle
from paper_2402_02082_gb300 import binding as gb
from paper_2402_02082_gb300 import build, synth

from gpu_util import assert_attn_close, dev, sample_pairs

pytestmark = pytest.mark.gpu

# Two fp32 evaluations of the same softmax average of values of order 1: each
# sums at most ~130 tiles a warp, 16 keys a tile and 64 warps, one rounding of
# 2^-24 a step, so either is within (130 + 16 + 64) 2^-24 = 1.3e-5 of exact.
AGREE = 2.6e-5


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gb.lib()


@pytest.mark.parametrize("B,H,D,dtype,kv,cap", [
    (1, 2, 128, "bf16", [1], 1),                 # one key, a cache of one row
    (2, 3, 128, "bf16", [15, 17], 17),           # around one tile; the cache ends with the keys
    (1, 32, 128, "bf16", [1023], 1024),          # clusters of 8, a ragged last tile
    (1, 32, 128, "bf16", [1025], 1100),          # one key into a second round
    (3, 32, 128, "bf16", [700, 1, 0], 704),      # clusters of 2, an empty sequence
    (4, 40, 64, "bf16", [129, 128, 127, 5], 130),
    (8, 40, 64, "bf16", [300, 31, 33, 0, 64, 65, 1, 299], 300),  # more (b, h) than a wave holds
    (8, 39, 64, "bf16", [2100] + [90] * 7, 2100),  # a thin second wave: clusters of 2
    (1, 12, 128, "bf16", [8500], 8512),          # long: clusters of 8 over many rounds
    (2, 200, 64, "bf16", [4100, 33], 4112),      # more than a wave and long: clusters of 4
    (1, 3, 64, "bf16", [8300], 8304),            # few heads, long: the streaming kernel
    (1, 4, 64, "f32", [128], 133),
    (2, 4, 128, "f32", [1000, 77], 1024),
    (1, 16, 128, "f32", [2100], 2112),           # fp32 clusters of 8: the streaming kernel
])
def test_cross_paths_agree(B, H, D, dtype, kv, cap):
    K = synth.normal_values(300 + cap, 1, (B, H, cap, D), dtype)
    V = synth.normal_values(300 + cap, 2, (B, H, cap, D), dtype)
    q = synth.normal_values(300 + cap, 3, (B, 1, H, D), dtype)
    nan = synth.BF16_NAN if dtype == "bf16" else np.float32(np.nan)
    for b, n in enumerate(kv):  # rows past the keys are never read
        K[b, :, n:] = nan
        V[b, :, n:] = nan
    desc = gb.make_desc(B, H, D, cap, gb.GLIDE_BF16 if dtype == "bf16" else gb.GLIDE_F32)
    ws = torch.zeros(gb.glide_attn_workspace_bytes(desc, 1), dtype=torch.uint8, device="cuda")
    qd, Kd, Vd, kvd = dev(q), dev(K), dev(V), dev(np.asarray(kv, np.int32))

    def run(max_ctas):
        out = torch.full((B, 1, H, D), float("nan"), device="cuda")
        gb.glide_cross_attn(qd, Kd, Vd, kvd, max(kv), out, ws, max_ctas=max_ctas)
        torch.cuda.synchronize()
        return out.cpu().numpy()

    auto, again, streaming = run(0), run(0), run(1)
    assert gb.glide_read_device_status(ws) == gb.GLIDE_OK
    for b, n in enumerate(kv):
        if n == 0:
            assert np.all(auto[b] == 0.0) and np.all(streaming[b] == 0.0)
    assert np.isfinite(auto).all()
    assert np.abs(auto - streaming).max() <= AGREE
    if max(kv) <= 8192 and not (dtype == "f32" and max(kv) > 2048):
        assert np.array_equal(auto, again), "fixed order of sums"
    pairs = [p for p in sample_pairs(B, H, 24, seed=3) if kv[p[0]] > 0]
    want = np.zeros((B, 1, H, D))
    for b, h in pairs:
        want[b, 0, h] = oracle.cross_attn(q[b:b + 1, :, h:h + 1], K[b:b + 1, h:h + 1], V[b:b + 1, h:h + 1], [kv[b]])[0, 0, 0]
    assert_attn_close(auto, want, pairs, f"cross B{B} H{H} D{D} {dtype} {kv}")


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_non_finite_scores(dtype):
    """The direct kernel: a NaN in a key is in its head's output and no other's; keys of score -inf have weight zero,
    a warp's whole tiles of them too."""
    B, H, D, n = 2, 4, 64, 300
    K = synth.normal_values(31, 1, (B, H, n, D), dtype)
    V = synth.normal_values(31, 2, (B, H, n, D), dtype)
    q = synth.normal_values(31, 3, (B, 1, H, D), dtype)
    qd, Kd, Vd, kvd = dev(q), dev(K), dev(V), dev(np.asarray([n, n], np.int32))
    qd[:, :, 1, 0] = 1.0
    keep = np.r_[0:16, 80:n]
    want = oracle.cross_attn(qd.float().cpu().numpy()[:1, :, 1:2], Kd.float().cpu().numpy()[:1, 1:2, keep],
                             Vd.float().cpu().numpy()[:1, 1:2, keep], [len(keep)])[0, 0, 0]
    Kd[0, 1, 16:80, 0] = float("-inf")
    Kd[1, 2, 37, 3] = float("nan")
    desc = gb.make_desc(B, H, D, n, gb.GLIDE_BF16 if dtype == "bf16" else gb.GLIDE_F32)
    ws = torch.zeros(gb.glide_attn_workspace_bytes(desc, 1), dtype=torch.uint8, device="cuda")
    out = torch.zeros((B, 1, H, D), device="cuda")
    gb.glide_cross_attn(qd, Kd, Vd, kvd, n, out, ws)
    got = out.cpu().numpy()
    nan = np.isnan(got).all(-1)[:, 0]
    assert nan.sum() == 1 and nan[1, 2] and np.isfinite(got[~nan[:, None]]).all()
    assert np.abs(got[0, 0, 1] - want).max() <= AGREE
