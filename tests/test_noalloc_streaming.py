"""glide_cross_attn_noalloc where a call does use the library's fixed array: the streaming kernel (few heads over a
long cache, and a bound on the CTAs below the direct kernel's) and the general grouped-query kernel, one call after
another, each with another layout of the array than the one before."""
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


def _case(B, H, H_kv, D, dtype, kv, max_ctas, seed):
    cap = max(kv)
    K = synth.normal_values(seed, 1, (B, H_kv, cap, D), dtype)
    V = synth.normal_values(seed, 2, (B, H_kv, cap, D), dtype)
    Kd, Vd, kvd = dev(K), dev(V), dev(np.asarray(kv, np.int32))

    def call(step):
        q = synth.normal_values(seed + 10 + step, 3, (B, 1, H, D), dtype)
        out = torch.full((B, 1, H, D), float("nan"), device="cuda")
        gb.glide_cross_attn_noalloc(dev(q), Kd, Vd, kvd, cap, out, max_ctas=max_ctas)
        assert gb.glide_noalloc_read_device_status() == gb.GLIDE_OK
        assert_attn_close(out.cpu().numpy(), oracle.cross_attn(q, K, V, kv), None, f"{B} {H}/{H_kv} {D} {dtype} {step}")

    return call


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
def test_layouts_in_turn(dtype):
    cases = [_case(1, 3, 3, 64, dtype, [8300], 0, 40),           # few heads, long: the streaming kernel
             _case(2, 8, 8, 128, dtype, [700, 33], 5, 41),       # a bound below the direct kernel's CTAs
             _case(1, 4, 2, 128, dtype, [1025], 3, 42),          # grouped queries, few CTAs: partials near the start
             _case(8, 32, 8, 64, dtype, [300, 1, 0, 64, 65, 299, 128, 17], 7, 43)]  # counters where those lay
    for step in range(2):
        for call in cases:
            call(step)
