"""The vocabulary argmax of greedy acceptance where rows do not start on 16-byte boundaries: a bulk
copy takes the floats between two boundaries, the ones of the row before are masked and the ones
past the last boundary loaded apart.  Trees of one node give each row's argmax as the bonus token."""
import numpy as np
import pytest
import torch

from paper_2402_02082_gb300 import binding as gb
from paper_2402_02082_gb300 import build

from gpu_util import dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    gb.lib()


def _argmax(logits):
    B, V = logits.shape
    i32 = dict(dtype=torch.int32, device="cuda")
    path, length, bonus = torch.full((B, 1), -5, **i32), torch.full((B,), -5, **i32), torch.full((B,), -5, **i32)
    ws = torch.zeros(gb.glide_accept_workspace_bytes(B, 1), dtype=torch.uint8, device="cuda")
    gb.tree_accept(torch.zeros((B, 1), **i32), torch.full((B, 1), -1, **i32), dev(logits[:, None]), path, length,
                   bonus, ws)
    torch.cuda.synchronize()
    assert gb.glide_read_device_status(ws) == gb.GLIDE_OK
    assert not path.any() and not length.any()
    return bonus.cpu().numpy()


@pytest.mark.parametrize("V", [1, 2, 3, 4, 5, 6, 7, 9, 127, 129, 4093, 4094, 4095, 4096, 4097, 4098, 4099, 8191, 8195,
                               12289, 32001])
def test_rows_of_any_length(V):
    B = 41
    rng = np.random.default_rng(V)
    x = rng.standard_normal((B, V)).astype(np.float32)
    # the maximum at a row's ends and around the chunks' ends, the neighbouring row's end larger still
    spots = sorted({min(V - 1, s) for s in (0, 1, 2, 3, V - 4, V - 3, V - 2, V - 1, 4092, 4094, 4095, 4096, 4097, 4099)
                    if s >= 0})
    for b in range(24):
        x[b, spots[b % len(spots)]] = 10.0 + b % 3
    x[24:28] = -np.inf                                  # no value at all: index 0
    x[28:32] = 1.5                                      # ties: the lowest index
    x[32, :] = -np.inf
    x[32, V - 1] = -1e30                                # the last float alone
    x[33], x[33, :V // 2 + 1] = 0.0, -0.0               # equal zeros
    assert np.array_equal(_argmax(x), x.argmax(-1))
