"""Calls whose outputs, lengths or parents do not lie as the kernels read and write them (dense rows
behind the pointer) are refused before the C call, by the binding's C++ marshalling and by its Python
code alike."""
import pytest
import torch

from paper_2402_02082_gb300 import binding as gb

B, H, D, CAP, N = 2, 4, 64, 96, 5


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2402_02082_gb300 import build
    build.build()


def _args(device):
    """C++ function -> (the binding's function, arguments by position, places of out, lengths, parents)"""
    def i32(v):
        return torch.tensor(v, dtype=torch.int32, device=device)

    K, V = (torch.zeros((B, H, CAP, D), device=device) for _ in range(2))
    q = {r: torch.zeros((B, r, H, D), device=device) for r in (1, N, CAP)}
    lens, parent = i32([70, 33]), i32([[-1, 0, 1, 1, 0]] * B)
    size = gb.glide_attn_workspace_bytes(gb.make_desc(B, H, D, CAP, gb.GLIDE_F32), N)
    ws = torch.zeros(size, dtype=torch.uint8, device=device)
    tail = (0.0, 0, 0, None)
    return {
        "cross_attn": (gb.glide_cross_attn, [q[1], K, V, lens, 70, q[1].clone(), ws, *tail], 5, 3, None),
        "cross_attn_noalloc": (gb.glide_cross_attn_noalloc, [q[1], K, V, lens, 70, q[1].clone(), *tail], 5, 3, None),
        "verify_attn": (gb.tree_verify_attn, [q[N], parent, K, V, lens, 70, q[N].clone(), ws, *tail], 6, 4, 1),
        "block_attn": (gb.glide_block_cross_attn, [q[CAP], K, V, lens, 5, q[CAP].clone(), ws, 0.0, 0, None], 5, 3, None),
    }


def _bad(args, out, lens, parent):
    """(place, argument) of the layouts that the kernels cannot use."""
    o, n = args[out], args[lens]
    yield out, o[:, :, :1].expand_as(o)                                        # every head's rows in one place
    yield out, o.transpose(2, 3).contiguous().transpose(2, 3)                  # right shape, other order
    yield out, torch.zeros((*o.shape[:-1], 2 * D), device=o.device)[..., :D]   # gaps between the rows
    yield lens, n[:-1]                                                         # a sequence without a length
    yield lens, n[:1].expand(B)
    yield lens, torch.stack([n, n], 1)[:, 0]
    if parent is not None:
        p = args[parent]
        yield parent, p.t().contiguous().t()
        yield parent, p[:1].expand(B, N)


NAMES = ["cross_attn", "cross_attn_noalloc", "verify_attn", "block_attn"]


@pytest.mark.parametrize("name", NAMES)
def test_refused_by_python(name):
    """Host tensors, which the C++ code leaves to Python: the refusal comes before any launch."""
    f, args, *places = _args("cpu")[name]
    for i, x in _bad(args, *places):
        with pytest.raises((TypeError, ValueError)):
            f(*args[:i], x, *args[i + 1:])


@pytest.mark.gpu
@pytest.mark.parametrize("name", NAMES)
def test_refused_with_device_tensors(name):
    f, args, *places = _args("cuda")[name]
    if name == "block_attn":
        args[:3] = [t.bfloat16() for t in args[:3]]
    native = getattr(gb._native(), name)
    for i, x in _bad(args, *places):
        bad = [*args[:i], x, *args[i + 1:]]
        assert native(*bad) == -1
        with pytest.raises((TypeError, ValueError)):
            f(*bad)


@pytest.mark.gpu
@pytest.mark.parametrize("name", NAMES[:3])
def test_longer_lengths_are_taken(name):
    """The lengths may be the start of a larger buffer, of any shape."""
    f, args, _, lens, _ = _args("cuda")[name]
    n = args[lens]
    for x in (torch.cat([n, n]), n[:, None]):
        assert getattr(gb._native(), name)(*args[:lens], x, *args[lens + 1:]) == gb.GLIDE_OK
    torch.cuda.synchronize()
