"""How multi-head cross-attention is split (csrc/cross_direct.cu): the CTAs per (sequence, head), on the
host with the runtime faked, and on the GPU the results of splits that do not divide the head size."""
import math
import os
import subprocess

import pytest
import torch

from paper_2402_02082_gb300 import binding as gb
from paper_2402_02082_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))
SLOTS = 304  # CTAs of the bf16 kernel that run at once on 152 SMs

# (B, H, D, fp32, keys) whose split has a remainder of head dims: 3, 5 and 6 CTAs
UNEVEN = [(5, 16, 64, 0, 700, 3), (5, 16, 128, 0, 600, 3), (2, 24, 64, 0, 2048, 5), (2, 24, 128, 0, 2049, 5),
          (1, 4, 64, 0, 700, 6), (1, 4, 128, 0, 655, 6), (1, 4, 64, 1, 700, 6), (2, 4, 128, 1, 641, 6),
          (2, 24, 64, 1, 2048, 5), (5, 16, 64, 1, 700, 3)]


@pytest.fixture(scope="module")
def split(tmp_path_factory):
    exe = str(tmp_path_factory.mktemp("split") / "check")
    cmd = [build.nvcc(), "-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-O0",
           "--expt-relaxed-constexpr", "-I", build.CSRC, "-I", build.INCLUDE, "-I", HERE,
           os.path.join(HERE, "cross_split_check.cu"), "-o", exe]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr

    def ask(shapes):
        lines = "\n".join(" ".join(str(x) for x in (*s, 0)[:6]) for s in shapes)
        r = subprocess.run([exe], input=lines, capture_output=True, text=True, timeout=60)
        assert r.returncode == 0
        out = [int(x) for x in r.stdout.split()]
        assert len(out) == len(shapes)
        return out

    return ask


def test_one_wave_is_not_left_half_empty(split):
    """A batch of 152 to 192 (sequence, head) over long caches: one CTA each would fill 51 to 63% of one wave,
    and nothing would fill the slots that short sequences leave."""
    shapes = [(B, H, D, 0, keys) for B, H in ((3, 52), (4, 40), (5, 32), (6, 32))
              for D in (64, 128) for keys in (6000, 8000, 12000, 16384)]
    for s, C in zip(shapes, split(shapes)):
        assert C == 0 or s[0] * s[1] * C > 1.2 * SLOTS, (s, C)


def test_bounds(split):
    shapes = [(B, H, D, f32, keys) for B, H in ((1, 1), (1, 32), (3, 40), (8, 52), (64, 40)) for D in (64, 128)
              for f32 in (0, 1) for keys in (1, 16, 128, 129, 300, 1000, 1024, 8192, 8193, 1 << 20, (1 << 31) - 1)]
    for s, C in zip(shapes, split(shapes)):
        assert 0 <= C <= 8
        if C > 1:
            assert (C - 1) * 128 < s[4], (s, C)  # every CTA of a cluster has a tile of the longest cache
        if s[4] < 1024:
            assert C > 0
    # a bound on the CTAs below the split's is left to the streaming kernel
    assert split([(1, 32, 128, 0, 2048, 255), (1, 32, 128, 0, 2048, 256)]) == [0, 8]


def test_uneven_splits_are_taken(split):
    assert split([s[:5] for s in UNEVEN]) == [s[5] for s in UNEVEN]


# Two fp32 evaluations of the same softmax average of values of order 1: at most 40 online updates a warp, 16
# keys a tile, 8 warps and 6 CTAs, one rounding of 2^-24 each: either is within 70 2^-24 = 4.2e-6 of exact, and
# values reach ~4.5.
AGREE = 2 * 4.5 * 70 * 2.0 ** -24


@pytest.mark.gpu
@pytest.mark.parametrize("B,H,D,f32,keys,_", UNEVEN)
def test_uneven_splits_agree(B, H, D, f32, keys, _):
    gen = torch.Generator(device="cuda").manual_seed(keys)
    dtype = torch.float32 if f32 else torch.bfloat16
    cap = keys + 7
    K, V = (torch.randn((B, H, cap, D), generator=gen, device="cuda", dtype=dtype) for _ in range(2))
    q = torch.randn((B, 1, H, D), generator=gen, device="cuda", dtype=dtype)
    lens = [keys - 131 * b for b in range(B)]
    for b, n in enumerate(lens):  # rows past the keys are never read
        K[b, :, n:] = float("nan")
        V[b, :, n:] = float("nan")
    ws = torch.zeros(gb.glide_attn_workspace_bytes(gb.make_desc(B, H, D, cap, gb.GLIDE_F32 if f32 else gb.GLIDE_BF16), 1),
                     dtype=torch.uint8, device="cuda")
    n = torch.tensor(lens, dtype=torch.int32, device="cuda")

    def run(max_ctas):
        out = torch.full((B, 1, H, D), float("nan"), device="cuda")
        return gb.glide_cross_attn(q, K, V, n, keys, out, ws, max_ctas=max_ctas)

    got, again, streaming = run(0), run(0), run(1)
    assert torch.equal(got, again)
    for b, n_b in enumerate(lens):
        k, v = K[b, :, :n_b].double(), V[b, :, :n_b].double()
        w = torch.softmax(torch.einsum("hd,hnd->hn", q[b, 0].double(), k) / math.sqrt(D), -1)
        want = torch.einsum("hn,hnd->hd", w, v)
        assert (got[b, 0] - want).abs().max() <= AGREE
        assert (streaming[b, 0] - want).abs().max() <= AGREE
