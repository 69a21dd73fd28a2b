"""The binding's C++ marshalling (csrc/pycall.cpp) against its Python code: what it takes gives the
same result as the Python code gives for the same arguments, and what is unusual or wrong it leaves
to the Python code."""
import numpy as np
import pytest
import torch

from paper_2402_02082_gb300 import binding as gb

B, H, D, CAP, N, V, GAMMA = 2, 4, 64, 96, 5, 100, 3


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_2402_02082_gb300 import build
    build.build()


def _calls(device, dtype, H_kv):
    """name of the C++ function -> (the binding's function, its arguments by position, its outputs)"""
    gen = torch.Generator().manual_seed(3)

    def rnd(*shape, t=torch.float32):
        return torch.randn(shape, generator=gen).to(t).to(device)

    def i32(v):
        return torch.tensor(v, dtype=torch.int32, device=device)

    def ws(size):
        return torch.zeros(size, dtype=torch.uint8, device=device)

    K, Vc = rnd(B, H_kv, CAP, D, t=dtype), rnd(B, H_kv, CAP, D, t=dtype)
    lens, parent = i32([70, 33]), i32([[-1, 0, 1, 1, 0]] * B)
    code = gb.GLIDE_BF16 if dtype == torch.bfloat16 else gb.GLIDE_F32
    w = ws(gb.glide_attn_workspace_bytes(gb.make_desc(B, H, D, CAP, code, H_kv=H_kv), N))
    q1, qn, qt = (rnd(B, r, H, D, t=dtype) for r in (1, N, CAP))
    tail = (0.0, 0, 0, None)
    logits, probs = rnd(B, N, V), torch.softmax(rnd(B, GAMMA, V), -1)

    def out(*shape, t=torch.float32):
        return torch.zeros(shape, dtype=t, device=device)

    def ints(*shape):
        return out(*shape, t=torch.int32)

    def cross():
        o = out(B, 1, H, D)
        return gb.glide_cross_attn, (q1, K, Vc, lens, 70, o, w, *tail), (o,)

    def noalloc():
        o = out(B, 1, H, D)
        return gb.glide_cross_attn_noalloc, (q1, K, Vc, lens, 70, o, *tail), (o,)

    def verify():
        o = out(B, N, H, D)
        return gb.tree_verify_attn, (qn, parent, K, Vc, lens, 70, o, w, *tail), (o,)

    def block():
        o = out(B, CAP, H, D)
        size = gb.glide_block_attn_workspace_bytes(gb.make_desc(B, H, D, CAP, code, H_kv=H_kv), CAP)
        return gb.glide_block_cross_attn, (qt, K, Vc, i32([CAP, 50]), 5, o, ws(max(size, 64)), 0.0, 0, None), (o,)

    def accept():
        o = (ints(B, N), ints(B), ints(B))
        return gb.tree_accept, (i32([[3, 5, 7, 9, 11]] * B), parent, logits, *o,
                                ws(gb.glide_accept_workspace_bytes(B, N)), None), o

    def expand():
        o = (ints(B, 17), ints(B, 17), ints(B))
        conf = out(B, GAMMA)
        return gb.cape_expand, (probs, i32([1, 2]), 16, *o, ws(gb.glide_cape_workspace_bytes(B, GAMMA, V)), conf, -1,
                                None), (*o, conf)

    def compact():
        o = ints(B)
        k, v = K.clone(), Vc.clone()
        path = i32([[0, 2, 4, -1, -1], [0, 1, -1, -1, -1]])
        return gb.glide_kv_compact, (k, v, i32([60, 20]), path, i32([3, 2]), o, None), (k, v, o)

    def sample():
        o = (ints(B), ints(B))
        return gb.spec_sample_accept, (i32([[1, 2, 3], [4, 5, 6]]), probs, rnd(B, GAMMA + 1, V),
                                       torch.rand((B, GAMMA + 1), generator=gen).to(device), *o,
                                       ws(gb.glide_sample_workspace_bytes(B, GAMMA)), None), o

    return dict(cross_attn=cross, cross_attn_noalloc=noalloc, verify_attn=verify, block_attn=block, accept=accept,
                expand=expand, compact=compact, sample=sample)


NAMES = ["cross_attn", "cross_attn_noalloc", "verify_attn", "block_attn", "accept", "expand", "compact", "sample"]


class _Sub(torch.Tensor):
    pass


@pytest.mark.parametrize("name", NAMES)
def test_left_to_python_on_the_host(name):
    """Host tensors, a missing argument, and anything that is no tensor are not taken."""
    _, args, _ = _calls("cpu", torch.float32, H)[name]()
    fn = getattr(gb._native(), name)
    assert fn(*args) == -1
    assert fn(*args[:-1]) == -1
    assert fn(None, *args[1:]) == -1
    assert fn() == -1


@pytest.mark.gpu
@pytest.mark.parametrize("dtype, H_kv", [(torch.float32, H), (torch.bfloat16, H), (torch.bfloat16, H // 2)])
@pytest.mark.parametrize("name", NAMES)
def test_same_as_python(name, dtype, H_kv, monkeypatch):
    """Both ways of marshalling end in the same C call: same status, same bytes."""
    if name == "block_attn" and dtype == torch.float32:
        pytest.skip("bf16 only")

    class Nothing:
        def __getattr__(self, _):
            return lambda *a: -1

    native, got = gb._native(), []
    for module in (native, Nothing()):
        f, args, outs = _calls("cuda", dtype, H_kv)[name]()
        monkeypatch.setattr(gb, "_CALL", module)
        f(*args)
        torch.cuda.synchronize()
        got.append([o.cpu() for o in outs])
    for a, b in zip(*got):
        assert torch.equal(a, b)
    assert any(bool(a.any()) for a in got[0])
    monkeypatch.setattr(gb, "_CALL", native)
    # the three documented forms of a stream are taken, on that stream
    _, args, _ = _calls("cuda", dtype, H_kv)[name]()
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    for stream in (side, side.cuda_stream, None):
        assert getattr(native, name)(*args[:-1], stream) == gb.GLIDE_OK
    torch.cuda.synchronize()


@pytest.mark.gpu
@pytest.mark.parametrize("name", NAMES)
def test_unusual_calls_are_left_to_python(name):
    """One argument at a time made unusual: none of these reaches the C call from C++."""
    native = getattr(gb._native(), name)
    _, args, _ = _calls("cuda", torch.bfloat16, H)[name]()
    for i, a in enumerate(args):
        if isinstance(a, torch.Tensor):
            swaps = [a.cpu(), a.as_subclass(_Sub)]
            if a.dtype != torch.uint8:  # a workspace's type and shape are free
                swaps += [a.to(torch.float64)]
                if not (i == 4 and name.startswith("verify")) and not (i == 3 and name.startswith("cross")):
                    swaps += [a[:-1], a[None, None]]  # kv_len's shape is not looked at
                if a.dim() > 1 and name not in ("cross_attn", "cross_attn_noalloc", "verify_attn"):
                    swaps += [a.transpose(-1, -2).contiguous().transpose(-1, -2)]
        elif a is None:
            swaps = ["0", 1.5]
        else:
            swaps = [np.int32(a), True, "0"]
        for x in swaps:
            assert native(*args[:i], x, *args[i + 1:]) == -1, (name, i, type(x))
    if "cross" in name or "verify" in name:
        with pytest.raises(TypeError):
            gb._native().cross_attn(q=args[0])
    torch.cuda.synchronize()


@pytest.mark.gpu
def test_status_is_raised():
    f, args, _ = _calls("cuda", torch.bfloat16, H)["cross_attn"]()
    with pytest.raises(gb.GlideError) as e:
        f(*args[:4], CAP + 1, *args[5:])
    assert e.value.status == gb.GLIDE_ERR_INVALID
    with pytest.raises(AttributeError):
        f(*args[:6], None, *args[7:])
