"""CaPE expansion over vocabularies of more than 32 chunks of 2048 (65536 tokens), where a lane merges the lists
of chunks s, s + 32, s + 64, ...: the largest probabilities in the later lists, and exact ties between them."""
import numpy as np
import pytest

from paper_2402_02082_gb300 import build, synth
from paper_2402_02082_gb300 import binding as gb

from test_cape_kv import assert_cape_equal

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gb.lib()


@pytest.mark.parametrize("V", [65536, 65537, 128256, 133120, 151936])  # 32, 33, 63, 65 and 75 chunks
def test_random(V):
    probs = synth.draft_probs(V, 2, 3, V)
    assert_cape_equal(probs, synth.root_tokens(7, 2, V), 32, None, f"V{V}")


@pytest.mark.parametrize("V", [65544, 128256, 151936])
def test_best_in_the_later_lists(V):
    """Position 0: the eight best in one late chunk; 1: one in each of chunks s, s + 32, s + 64 (as far as V goes),
    equal in pairs, so that the lower token wins; 2: the last tokens of the vocabulary."""
    chunk, B, gamma = 2048, 2, 3
    probs = synth.draft_probs(V + 1, B, gamma, V).astype(np.float32) * np.float32(0.1)
    rng = np.random.default_rng(V)
    last = (V - 1) // chunk
    for b in range(B):
        at = last * chunk + rng.permutation(min(chunk, V - last * chunk))[:8]
        probs[b, 0, at] = np.float32(0.05) + np.float32(0.003) * np.arange(8, dtype=np.float32)
        s = int(rng.integers(last - 32 + 1)) if last >= 32 else 0
        for i, c in enumerate(range(s, last + 1, 32)):
            off = int(rng.integers(min(chunk, V - c * chunk)))
            probs[b, 1, c * chunk + off] = np.float32(0.2)
            probs[b, 1, c * chunk + (off + 7) % min(chunk, V - c * chunk)] = np.float32(0.1)
        probs[b, 2, V - 8:] = np.float32(0.04)
    assert_cape_equal(probs, synth.root_tokens(9, B, V), 32, None, f"V{V} late")
    assert_cape_equal(probs, synth.root_tokens(9, B, V), 63, 7, f"V{V} late, fixed size")
