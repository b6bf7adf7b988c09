"""Calls in a row, each on what the one before it wrote: the small launches are set up while their predecessor is still running, and
must not touch memory before it is complete.  The same calls, the device waited for after each, give the same bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

la = pytest.importorskip("paper_2509_24695_b200")

# tokens, heads, head dim, dtype, rotary: lone CTAs, clusters, the grid; fp32 as a cluster and with partial states; general kernels
SHAPES = [(64, 4, 32, "bf16", False), (192, 4, 32, "bf16", False), (300, 3, 112, "bf16", True), (1200, 4, 64, "bf16", True),
          (7000, 2, 112, "bf16", False), (96, 2, 128, "bf16", True), (150, 3, 112, "f32", False), (6000, 20, 64, "f32", True),
          (130, 5, 40, "bf16", False), (77, 3, 8, "f32", False)]


def chain(N, H, d, dtype, rope, wait, capture=False, rounds=6):
    dt = {"bf16": torch.bfloat16, "f32": torch.float32}[dtype]
    gen = torch.Generator(device="cuda").manual_seed(N * 131 + d)
    x = torch.randn(1, N, H, d, device="cuda", generator=gen).to(dt)
    w = torch.randn(3, H * d, device="cuda", generator=gen) * 0.25
    ang = torch.randn(N, d // 2, device="cuda", generator=gen)
    buf = [x.clone() for _ in range(3)]
    y = torch.zeros(1, 2, N, H * d, device="cuda", dtype=dt)
    tab = la.rope_pack(ang.cos(), ang.sin())
    cache = la.BlockLinCache(1, H, d, dt, "cuda", max_T_b=N)
    conv = la.TConvCache(1, N, H * d, dt, "cuda")
    ws = la.new_rope_workspace(x) if rope else la.new_workspace(x)
    torch.cuda.synchronize()

    def once():
        done = torch.cuda.synchronize if wait else (lambda: None)
        for r in range(rounds):
            a, b, c = buf[r % 3], buf[(r + 1) % 3], buf[(r + 2) % 3]
            # queries, keys and values written by the calls before; the output over what the call before last read
            if rope:
                la.linattn_forward_rope(a, b, a, tab, out=c, workspace=ws)
            else:
                la.linattn_forward(a, b, a, out=c, workspace=ws)
            done()
            o, p = y[:, 0].view(1, N, H, d), y[:, 1].view(1, N, H, d)
            cache.step_rope(c, a, b, tab, out=o) if rope else cache.step(c, a, b, out=o)
            done()
            cache.peek_rope(a, c, b, tab, out=p) if rope else cache.peek(a, c, b, out=p)
            done()
            z = conv.step(y, w)           # reads both outputs; keeps the second
            done()
            a.copy_((z[:, 1] * 4).view(1, N, H, d))   # a torch kernel in between
            done()
            la.linattn_state(z[:, 0].view(1, N, H, d), a, out=state, workspace=ws2)
            done()
            la.linattn_apply(a, state, out=b, workspace=ws2)
            done()

    ws2 = la.new_workspace(x)
    state = torch.empty(1, H, d + 1, d, device="cuda")
    if capture:
        s = torch.cuda.Stream()
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g, stream=s):
            once()
        g.replay()
    else:
        once()
    torch.cuda.synchronize()
    return [t.clone() for t in (*buf, y, state, cache.state, conv.frame)]


@pytest.mark.parametrize("shape", SHAPES, ids=str)
def test_calls_in_a_row(shape):
    want = chain(*shape, wait=True)
    assert all(t.isfinite().all() for t in want)
    for _ in range(3):
        for got, ref in zip(chain(*shape, wait=False), want):
            assert torch.equal(got, ref)


@pytest.mark.parametrize("shape", SHAPES[1::3], ids=str)
def test_calls_in_a_row_captured(shape):
    for got, ref in zip(chain(*shape, wait=False, capture=True), chain(*shape, wait=True)):
        assert torch.equal(got, ref)


@pytest.mark.parametrize("shape", [SHAPES[1], SHAPES[2], SHAPES[6]], ids=str)
def test_calls_behind_memsets_copies_and_joins(shape):
    """What stands before a call is not always a kernel of its stream: a memset, a copy, the join of two streams; eager and captured."""
    N, H, d, dtype, rope = shape
    dt = {"bf16": torch.bfloat16, "f32": torch.float32}[dtype]
    gen = torch.Generator(device="cuda").manual_seed(N + d)
    x0, x1 = (torch.randn(1, N, H, d, device="cuda", generator=gen).to(dt) for _ in range(2))
    w = torch.randn(3, H * d, device="cuda", generator=gen) * 0.25
    x, o, p, z = (torch.zeros_like(x0) for _ in range(4))
    cache, conv = la.BlockLinCache(1, H, d, dt, "cuda", max_T_b=N), la.TConvCache(1, N, H * d, dt, "cuda")
    ws = la.new_workspace(x)
    side = torch.cuda.Stream()

    def once(done=lambda: None):
        main = torch.cuda.current_stream()
        cache.reset()                                        # a memset
        cache.step(x1, x1, x0, out=o)
        done()
        x.copy_(o)                                           # a copy
        cache.peek(x, x1, x0, out=p)
        done()
        side.wait_stream(main)
        with torch.cuda.stream(side):
            conv.reset()
            conv.step(p.view(1, 1, N, H * d), w, out=z.view(1, 1, N, H * d))
        done()
        cache.step(p, x, x1, out=o)
        main.wait_stream(side)
        done()
        la.linattn_forward(z, o, x0, out=x, workspace=ws)    # behind both streams
        done()

    once(torch.cuda.synchronize)
    want = [t.clone() for t in (x, o, p, z, cache.state, conv.frame)]
    got = []
    once()
    torch.cuda.synchronize()
    got.append([t.clone() for t in (x, o, p, z, cache.state, conv.frame)])
    g, s = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(g, stream=s):
        once()
    for t in (x, o, p, z):
        t.zero_()
    for _ in range(2):
        g.replay()
        torch.cuda.synchronize()
        got.append([t.clone() for t in (x, o, p, z, cache.state, conv.frame)])
    for run in got:
        for a, b in zip(run, want):
            assert b.isfinite().all() and torch.equal(a, b)
