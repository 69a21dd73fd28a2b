"""Speculative-sampling acceptance where its split changes: the cluster sizes that different numbers
of sequences give, and vocabularies around a chunk of a row's part (16384 tokens), a segment's
32-token groups and the weights that stay in shared memory (32 x 1632 tokens)."""
import numpy as np
import pytest
import torch

from paper_2402_02082_gb300 import binding as gb
from paper_2402_02082_gb300 import build, synth

from test_sampling import compare, run

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gb.lib()


@pytest.mark.parametrize("B,gamma,V", [
    (1, 63, 33),        # more parts than any cluster has warps
    (1, 5, 16384), (2, 1, 16383), (3, 2, 16388), (2, 4, 32768), (1, 2, 32772), (2, 3, 16401),
    (1, 1, 1), (8, 1, 2), (15, 2, 31), (16, 6, 1000), (23, 2, 1025), (29, 1, 333), (37, 3, 64), (47, 2, 100),
    (77, 1, 512), (153, 1, 40),
    (2, 2, 52224), (2, 2, 52225), (1, 1, 70001),
])
def test_split_edges(B, gamma, V):
    q = synth.draft_probs(700 + V + gamma, B, gamma, V) if V > 1 else np.ones((B, gamma, 1), np.float32)
    draft = synth.sample_tokens(701 + V, q)
    logits = synth.target_logits_near(702 + V, q, 0.6) if V > 1 else np.zeros((B, gamma + 1, 1), np.float32)
    u = synth.uniforms(703 + V, (B, gamma + 1))
    n, t, ws = run(draft, q, logits, u)
    assert compare(draft, q, logits, u, n, t) <= 1
    again = run(draft, q, logits, u, ws)
    assert np.array_equal(n, again[0]) and np.array_equal(t, again[1])
