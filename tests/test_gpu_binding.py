"""The short way from torch tensors to the library (csrc/binding.cpp) against the general one: the same results, and whatever it does
not take ends where the general way ends."""
import ctypes
import types

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

la = pytest.importorskip("paper_2509_24695_b200")


def qkv(*shape, dtype=torch.bfloat16, head_major=False):
    gen = torch.Generator(device="cuda").manual_seed(5)
    B, N, H, d = shape
    return [torch.randn(B, H, N, d, device="cuda", generator=gen).to(dtype).permute(0, 2, 1, 3) if head_major
            else torch.randn(B, N, H, d, device="cuda", generator=gen).to(dtype) for _ in range(3)]


def calls(dtype=torch.bfloat16, head_major=False, out=False):
    """Every call that has a short way, from the same inputs."""
    B, N, H, d = 2, 70, 3, 112
    q, k, v = qkv(B, N, H, d, dtype=dtype, head_major=head_major)
    ang = torch.rand(N, d // 2, device="cuda", generator=torch.Generator(device="cuda").manual_seed(6))
    tab = la.rope_pack(ang.cos(), ang.sin())
    new = torch.empty_like if out else (lambda t: None)
    res = [la.linattn_forward(q, k, v, out=new(q), workspace=la.new_workspace(q)),
           la.linattn_forward(q, k, v, 1e-3, new(q), la.new_workspace(q)),
           la.linattn_forward_rope(q, k, v, tab, out=new(q), workspace=la.new_rope_workspace(q))]
    q, k, v = (t.contiguous() for t in (q, k, v))
    cache = la.BlockLinCache(B, H, d, dtype, "cuda", max_T_b=N)
    res += [cache.step(q, k, v, out=new(q)), cache.peek(q, v, k, out=new(q))]
    cache.reset()
    res += [cache.step_rope(q, k, v, tab, out=new(q)), cache.peek_rope(q, v, k, tab, out=new(q)), cache.state.clone()]
    assert cache.info() == {"blocks_seen": 1, "tokens_seen": N, "state_bytes": cache.state.numel() * 4}
    x = q.reshape(B, N // 5, 5, H * d)
    w = torch.randn(3, H * d, device="cuda", generator=torch.Generator(device="cuda").manual_seed(7))
    conv = la.TConvCache(B, 5, H * d, dtype, "cuda")
    res += [la.tconv_forward(x, w, out=new(x)), conv.step(x, w, out=new(x)), conv.step(x, w, commit=False), conv.frame.clone()]
    return res


@pytest.mark.parametrize("kw", [{}, {"dtype": torch.float32}, {"head_major": True}, {"out": True}], ids=str)
def test_both_ways(kw, monkeypatch):
    la._bind(la.load_library())
    assert la._fast is not la._NoBinding, "the binding is not built"
    got = calls(**kw)
    monkeypatch.setattr(la, "_fast", la._NoBinding)
    for a, b in zip(got, calls(**kw)):
        assert torch.equal(a, b) and a.stride() == b.stride() and not a.requires_grad


def test_out_is_returned_and_streams_are_followed():
    q, k, v = qkv(1, 500, 4, 64)
    ws, out = la.new_workspace(q), torch.empty_like(q)
    want = la.linattn_forward(q, k, v, workspace=ws)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    with torch.cuda.stream(s):
        big = torch.randn(4096, 4096, device="cuda")
        for _ in range(20):
            big = big @ big * 1e-4
        late = q + 0 * big[0, 0].nan_to_num(0.0).to(q.dtype)   # (ready long after the call is made)
        assert la.linattn_forward(late, k, v, out=out, workspace=ws) is out
    s.synchronize()
    assert torch.equal(out, want)


def test_what_is_not_plain_ends_as_before():
    q, k, v = qkv(1, 40, 2, 64)
    ws = la.new_workspace(q)
    want = la.linattn_forward(q, k, v, workspace=ws)
    with torch.inference_mode():
        assert torch.equal(la.linattn_forward(q, k, v, workspace=ws), want)
    assert torch.equal(la.linattn_forward(torch.nn.Parameter(q), k, v, workspace=ws), want)
    assert torch.equal(la.linattn_forward(q, k, v, eps=1e-6), want)        # no workspace
    for bad in ((q[:, :39], k, v), (q, k.float(), v), (q, k, v.cpu()), (q.cpu(), k.cpu(), v.cpu()), (q[0], k[0], v[0])):
        with pytest.raises(ValueError):
            la.linattn_forward(*bad, workspace=ws)
    with pytest.raises(TypeError):
        la.linattn_forward(q.half(), k.half(), v.half(), workspace=ws)
    with pytest.raises(la.LinAttnError):
        la.linattn_forward(q, k, v, out=q, workspace=ws)                   # over its input
    with pytest.raises(la.LinAttnError):
        la.linattn_forward(q, k, v, workspace=ws[:4096])
    with pytest.raises(RuntimeError):
        torch.vmap(lambda t: la.linattn_forward(t, k, v, workspace=ws))(torch.stack([q, q]))
    cache = la.BlockLinCache(1, 2, 64, torch.bfloat16, "cuda", max_T_b=40)
    with pytest.raises(ValueError):
        cache.step(q[..., :32], k[..., :32], v[..., :32])
    with pytest.raises(ValueError):
        cache.step(*(t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in (q, k, v)))   # dense blocks only
    cache.close()
    with pytest.raises(la.LinAttnError):
        cache.step(q, k, v)


def test_modes_see_the_allocation():
    """A torch function mode and a dispatch mode are asked, as they are the general way."""
    from torch.overrides import TorchFunctionMode
    from torch.utils._python_dispatch import TorchDispatchMode

    q, k, v = qkv(1, 40, 2, 64)
    ws, seen = la.new_workspace(q), []

    class Functions(TorchFunctionMode):
        def __torch_function__(self, func, types, args=(), kwargs=None):
            seen.append(func)
            return func(*args, **(kwargs or {}))

    class Dispatch(TorchDispatchMode):
        def __torch_dispatch__(self, func, types, args=(), kwargs=None):
            seen.append(func)
            return func(*args, **(kwargs or {}))

    for mode in (Functions, Dispatch):
        seen.clear()
        with mode():
            la.linattn_forward(q, k, v, workspace=ws)
        assert any("empty_like" in str(f) for f in seen)


@pytest.mark.parametrize("name", la._FAST_CALLS)
def test_a_failed_call_is_not_made_again(name, monkeypatch):
    """A call that commits a block may have done so before it failed (its second launch, say): one call to the library, one error.
    Stand-ins for the library's functions fail the first time only, so a second try would pass unseen; nothing is launched."""
    lib, made = la.load_library(), []

    def fails_once(*args):
        made.append(name)
        return -5 if len(made) == 1 else 0

    callback = ctypes.CFUNCTYPE(ctypes.c_int, *(t if isinstance(t, type) and issubclass(t, ctypes._SimpleCData) else ctypes.c_void_p
                                                for t in getattr(lib, name).argtypes))(fails_once)
    stand_in = types.SimpleNamespace(**{n: callback if n == name else getattr(lib, n) for n in la._FAST_CALLS})
    q, k, v = qkv(1, 40, 2, 64)
    tab = torch.zeros(40, 32, 2, dtype=torch.float16, device="cuda")
    x, w = q.view(1, 4, 10, 128), torch.zeros(3, 128, device="cuda")
    cache = la.BlockLinCache(1, 2, 64, torch.bfloat16, "cuda", max_T_b=40)
    conv = la.TConvCache(1, 10, 128, torch.bfloat16, "cuda")
    ws, rope_ws = la.new_workspace(q), la.new_rope_workspace(q)
    call = {"linattn_forward": lambda: la.linattn_forward(q, k, v, workspace=ws),
            "linattn_forward_rope": lambda: la.linattn_forward_rope(q, k, v, tab, workspace=rope_ws),
            "blocklin_step": lambda: cache.step(q, k, v), "blocklin_peek": lambda: cache.peek(q, k, v),
            "blocklin_step_rope": lambda: cache.step_rope(q, k, v, tab), "blocklin_peek_rope": lambda: cache.peek_rope(q, k, v, tab),
            "tconv_forward": lambda: la.tconv_forward(x, w), "tconv_block_step": lambda: conv.step(x, w)}[name]
    monkeypatch.setattr(lib, name, fails_once)   # (for the general way)
    try:
        la._bind(stand_in)
        assert la._fast is not la._NoBinding, "the binding is not built"
        with pytest.raises(la.LinAttnError, match=f"^{name}: .*status -5"):
            call()
        assert made == [name]
        assert call() is not None and made == [name, name]   # (and the next call is a call like any other)
    finally:
        monkeypatch.undo()
        la._bind(lib)


@pytest.mark.parametrize("which", ["q", "k", "v", "out", "table", "ws", "x", "w", "frame"])
def test_a_pointer_that_cannot_be_had_is_an_error(which):
    """Memory that throws when it is asked for (here because it is told to) ends in Python's error, as the general way."""
    q, k, v = qkv(1, 40, 2, 64)
    t = {"q": q, "k": k, "v": v, "out": torch.empty_like(q), "table": torch.zeros(40, 32, 2, dtype=torch.float16, device="cuda"),
         "ws": la.new_rope_workspace(q), "x": q.clone().view(1, 4, 10, 128), "w": torch.zeros(3, 128, device="cuda")}
    conv = la.TConvCache(1, 10, 128, torch.bfloat16, "cuda")
    cache = la.BlockLinCache(1, 2, 64, torch.bfloat16, "cuda", max_T_b=40)
    t["frame"] = conv.frame
    calls = {"attention": [lambda: la.linattn_forward(t["q"], t["k"], t["v"], out=t["out"], workspace=t["ws"]),
                           lambda: la.linattn_forward_rope(t["q"], t["k"], t["v"], t["table"], out=t["out"], workspace=t["ws"]),
                           lambda: cache.step(t["q"], t["k"], t["v"], out=t["out"]),
                           lambda: cache.peek_rope(t["q"], t["k"], t["v"], t["table"], out=t["out"])],
             "conv": [lambda: la.tconv_forward(t["x"], t["w"]), lambda: conv.step(t["x"], t["w"])]}
    takes = {"table": [1, 3], "ws": [0, 1], "frame": [1]}.get(which, range(4))
    torch._C._set_throw_on_mutable_data_ptr(t[which])
    for i, call in enumerate(calls["conv" if which in ("x", "w", "frame") else "attention"]):
        if i in takes:
            with pytest.raises(RuntimeError, match="data pointer"):
                call()
        else:
            call()
    torch.cuda.synchronize()
