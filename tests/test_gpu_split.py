"""The fp32-accurate path (fp32 tensors, bf16 head dims outside the fused kernel's) at the edges of its tiles: every
padding class of the head dim, token counts around the staged tiles and the split over CTAs, and the general kernels it
shares the path with (rows that cannot be read in 16-byte pieces)."""
import numpy as np
import pytest

import synth
from parity_util import assert_parity_bf16, assert_parity_f32, assert_state_close, to_dev, to_f64

pytestmark = pytest.mark.gpu

EPS = 1e-6
HEAD_DIMS = {"f32": [4, 12, 32, 36, 64, 80, 84, 100, 112, 116, 128], "bf16": [8, 24, 40, 56, 72, 88, 96, 104, 120]}


@pytest.fixture(scope="module")
def la():
    import torch

    assert torch.cuda.is_available(), "these tests need a CUDA device"
    import paper_2509_24695_b200 as la

    la.load_library()
    return la


def gen(B, N, H, d, seed, dtype):
    return tuple(synth.gauss((B, N, H, d), seed, t, dtype=dtype) for t in (1, 2, 3))


def check(dtype, got, ref, what):
    (assert_parity_bf16 if dtype == "bf16" else assert_parity_f32)(got, ref, what)


@pytest.mark.parametrize("dtype,d", [(t, d) for t in HEAD_DIMS for d in HEAD_DIMS[t]])
@pytest.mark.parametrize("N", [1, 33, 127, 1300])
def test_tiles(la, orc, dtype, d, N):
    B, H = 2, 3
    q, k, v = gen(B, N, H, d, 7000 + N + d, dtype)
    S, z = orc.state(k, v)
    st = la.linattn_state(to_dev(k), to_dev(v))
    assert_state_close(to_f64(st), S, z, 1e-5, f"state N={N} d={d} {dtype}")
    o = la.linattn_forward(to_dev(q), to_dev(k), to_dev(v), EPS)
    check(dtype, to_f64(o), orc.forward(q, k, v, EPS), f"forward N={N} d={d} {dtype}")
    cos, sin = synth.rope_table(1, 1, N, d)
    table = la.rope_pack(to_dev(cos), to_dev(sin))
    packed = table.cpu().numpy().astype(np.float64)
    o = la.linattn_forward_rope(to_dev(q), to_dev(k), to_dev(v), table, EPS)
    check(dtype, to_f64(o), orc.rope_forward(q, k, v, packed[..., 0], packed[..., 1], EPS), f"rotary N={N} d={d} {dtype}")


@pytest.mark.parametrize("dtype,d", [("f32", 112), ("f32", 64), ("bf16", 72)])
def test_rows_off_the_16_byte_grid(la, orc, dtype, d):
    """The same values one element further in memory, with head and token strides that are no multiple of 16 bytes,
    and head-major."""
    import torch

    B, N, H = 1, 700, 3
    q, k, v = gen(B, N, H, d, 7100 + d, dtype)
    ref = orc.forward(q, k, v, EPS)

    def shifted(x):
        t = to_dev(x)
        flat = torch.empty(t.numel() + 1, dtype=t.dtype, device="cuda")
        flat[1:] = t.flatten()
        return flat[1:].view(t.shape)

    def strided(x):
        t = torch.zeros((B, N, H, d + 1), dtype=to_dev(x).dtype, device="cuda")[..., :d]
        return t.copy_(to_dev(x))

    def head_major(x):
        return to_dev(x).permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3)

    for place in (shifted, strided, head_major):
        o = la.linattn_forward(place(q), place(k), place(v), EPS, out=place(q))
        check(dtype, to_f64(o), ref, f"{place.__name__} {dtype} d={d}")
    # an output off the grid beside inputs on it
    out = shifted(q) if dtype == "f32" else None
    if out is not None:
        o = la.linattn_forward(to_dev(q), to_dev(k), to_dev(v), EPS, out=out)
        check(dtype, to_f64(o), ref, "shifted output")


@pytest.mark.parametrize("dtype,d,N", [("f32", 112, 5000), ("bf16", 72, 9000), ("f32", 64, 200), ("bf16", 96, 700)])
def test_cached_step_and_its_read_only_twin(la, orc, dtype, d, N):
    """On top of an old state, with the CTAs of a unit as a cluster (few tokens) and with partial states (many)."""
    import torch

    B, H = 1, 3
    q, k, v = gen(B, N, H, d, 7200 + N, dtype)
    k0, v0 = gen(B, 50, H, d, 7300 + N, dtype)[1:]
    td = torch.float32 if dtype == "f32" else torch.bfloat16
    cache = la.BlockLinCache(B, H, d, td, "cuda", max_T_b=N, eps=EPS)
    cache.step(None, to_dev(k0), to_dev(v0))
    before = cache.state.clone()
    o_peek = cache.peek(to_dev(q), to_dev(k), to_dev(v))
    assert torch.equal(cache.state, before)
    o = cache.step(to_dev(q), to_dev(k), to_dev(v))
    assert torch.equal(o, o_peek) and cache.status() == 0
    (S0, z0), (S, z) = orc.state(k0, v0), orc.state(k, v)
    assert_state_close(to_f64(cache.state), S0 + S, z0 + z, 1e-5, f"cache N={N} d={d} {dtype}")
    ref = orc.apply_rows(q, S0 + S, z0 + z, EPS, np.arange(N))
    check(dtype, to_f64(o), ref, f"step N={N} d={d} {dtype}")


def turned(x, table):
    """Feature pairs of x[B, N, H, d] turned by the (cos, sin) of their token, table [N, d/2, 2]."""
    if table is None:
        return x
    c, s = table[None, :, None, :, 0], table[None, :, None, :, 1]
    a, b = x[..., 0::2], x[..., 1::2]
    return np.stack((a * c - b * s, b * c + a * s), axis=-1).reshape(x.shape)


def relative(got, ref):
    return np.sqrt(((got - ref) ** 2).sum() / (ref ** 2).sum())


@pytest.mark.parametrize("dtype,d,rope", [("f32", 112, False), ("f32", 24, False), ("f32", 64, True), ("bf16", 72, True),
                                          ("bf16", 40, False)])
@pytest.mark.parametrize("N", [1, 50, 1500])
def test_infinite_values(la, dtype, d, rope, N):
    """One infinite value gives infinities in its column of S (and of the outputs, where no two of them meet), as a sum of
    products does, and nothing anywhere else."""
    import torch

    B, H, j = 1, 3, 5
    q, k, v = (to_dev(x) for x in gen(B, N, H, d, 7400 + N + d, dtype))
    q, k = q.abs() + 0.125, k.abs() + 0.125          # every product with the infinity is one
    v[0, N // 2, 1, j] = float("inf")
    table = None
    if rope:
        cos, sin = synth.rope_table(1, 1, N, d)
        table = la.rope_pack(to_dev(cos), to_dev(sin))
    tab = None if table is None else table.cpu().numpy().astype(np.float64)
    qn, kn, vn = to_f64(q), to_f64(k), to_f64(v)
    kt, qt = turned(kn, tab), turned(qn, tab)
    with np.errstate(invalid="ignore"):
        S = np.einsum("bnhi,bnhj->bhij", kt, vn)
        O = np.einsum("bnhi,bhij->bnhj", qt, S) / (np.einsum("bnhi,bhi->bnh", qn, kn.sum(1)) + EPS)[..., None]
    if rope:
        cache = la.BlockLinCache(B, H, d, q.dtype, "cuda", max_T_b=N, eps=EPS)
        o, st = cache.step_rope(q, k, v, table), cache.state
    else:
        o, st = la.linattn_forward(q, k, v, EPS), la.linattn_state(k, v)
    for got, ref, bar in ((to_f64(st)[:, :, :d].swapaxes(-1, -2), S, 1e-5), (to_f64(o), O, 1e-5 if dtype == "f32" else 1e-2)):
        finite = np.isfinite(ref)
        assert not finite[..., 1, :, j].any() if got.shape == S.shape else not finite[:, :, 1, j].any()
        assert np.array_equal(got[~finite], ref[~finite], equal_nan=True)
        assert np.isfinite(got[finite]).all() and relative(got[finite], ref[finite]) <= bar


@pytest.mark.parametrize("d", [24, 64, 112])
@pytest.mark.parametrize("tensor,scale", [("k", 1e-35), ("v", 1e-36), ("q", 1e-35), ("v", 1e-41), ("kv", 1e-19), ("v", 3e38)])
def test_tiny_and_huge_values(la, d, tensor, scale):
    """Values whose low bits no bf16 holds, subnormal ones, sums around the smallest normal number, values next to the largest
    one.  Bar: a chain of fp32 multiply-adds rounds by up to 2^-24 a step (300 of them, random signs: 5e-7), and by 2^-149 where
    sums are subnormal (around 1e-41)."""
    import torch

    B, N, H = 1, 300, 3
    x = dict(zip("qkv", (to_dev(t) for t in gen(B, N, H, d, 7500 + d, "f32"))))
    x["q"], x["k"] = x["q"].abs(), x["k"].abs()
    if scale > 1:   # one term to a sum: half of |v| up to 3.4e38, no overflow
        x["k"].zero_()
        x["k"][:, -1] = 0.5
        x["v"] = x["v"].clamp(-1, 1) * 3.4028e38
        x["q"] = torch.full_like(x["q"], 1.0 / d)
    else:
        for name in tensor:
            x[name] = x[name] * scale
    q, k, v = (x[n] for n in "qkv")
    qn, kn, vn = to_f64(q), to_f64(k), to_f64(v)
    S, z = np.einsum("bnhi,bnhj->bhij", kn, vn), kn.sum(1)
    bar = max(2e-6, 300 * 2.0 ** -149 / np.sqrt((S ** 2).mean()))
    st = la.linattn_state(k, v)
    assert relative(to_f64(st)[:, :, :d].swapaxes(-1, -2), S) <= bar
    num = np.einsum("bnhi,bhij->bnhj", qn, to_f64(st)[:, :, :d].swapaxes(-1, -2))
    O = num / (np.einsum("bnhi,bhi->bnh", qn, z) + EPS)[..., None]
    bar = max(2e-6, 2.0 ** -149 * (d / np.sqrt((num ** 2).mean()) + 1 / np.sqrt((O ** 2).mean())))
    assert relative(to_f64(la.linattn_apply(q, st, EPS)), O) <= bar


def spread(kind, shape, seed):
    """Inputs on which products of parts could lose more than a multiply-add rounds: constants whose second and third parts
    are as large as they get, values of one sign, log-normal and normal ones."""
    if kind.startswith("constant"):
        value = {"constant_cut": 1 + 2.0 ** -7 - 2.0 ** -23, "constant_rounded": 1 + 2.0 ** -8 - 2.0 ** -17, "constant_third": 1 / 3}[kind]
        return tuple(np.full(shape, value, dtype=np.float32) for _ in range(3))
    x = tuple(synth.gauss(shape, seed, t, dtype="f32") for t in (1, 2, 3))
    return x if kind == "normal" else tuple(np.abs(t) + 1 for t in x) if kind == "one_sign" else tuple(np.exp(t) for t in x)


@pytest.mark.parametrize("kind", ["constant_cut", "constant_rounded", "constant_third", "one_sign", "log_normal", "normal"])
@pytest.mark.parametrize("d", [32, 112])
def test_no_further_from_64_bits_than_multiply_adds(la, kind, d):
    """Bars on the 2-norm of S and z.  One token: a product rounded to nearest, 2^-24.  More: up to 2^-24 for the products left
    out, 2^-24 for each of the few sums in registers, random signs: 2^-22.  (Six products of parts cut off: 2^-21 alone.)  O on
    top of the rounded state: 112 products and a quotient, 2^-21."""
    for N in (1, 2, 7, 32, 64, 65, 200, 512):
        q, k, v = spread(kind, (1, N, 3, d), 7600 + N)
        qn, kn, vn = (x.astype(np.float64) for x in (q, k, v))
        qn, kn = qn.clip(0), kn.clip(0)
        st = to_f64(la.linattn_state(to_dev(k), to_dev(v)))
        S, z = np.einsum("bnhi,bnhj->bhji", kn, vn), kn.sum(1)
        bar = 1.01 * 2.0 ** -24 if N == 1 else 2.0 ** -22
        assert relative(st[:, :, :d], S) <= bar, f"S, {N} tokens: {relative(st[:, :, :d], S):.2e}"
        assert relative(st[:, :, d], z) <= bar, f"z, {N} tokens"
        O = np.einsum("bnhi,bhji->bnhj", qn, S) / (np.einsum("bnhi,bhi->bnh", qn, z) + EPS)[..., None]
        o = to_f64(la.linattn_forward(to_dev(q), to_dev(k), to_dev(v), EPS))
        assert relative(o, O) <= 2.0 ** -21, f"O, {N} tokens: {relative(o, O):.2e}"


def test_a_state_is_held_back_for_its_own_launch_alone(la):
    """A state stays as it was when a CTA of its own launch gave up (said so in the second word of the control block), and only
    then: not because the status word still has a timeout from before."""
    import torch

    q, k, v = (to_dev(x) for x in gen(1, 6000, 20, 112, 7700, "f32"))
    want = la.linattn_state(k, v)
    ws = la.new_workspace(k)
    words = ws[:16].view(torch.int32)
    out = torch.full_like(want, 7.0)
    before = la.load_library().linattn_kernel_launches()
    words[1] = 1
    la.linattn_state(k, v, out=out, workspace=ws)
    assert la.load_library().linattn_kernel_launches() == before + 2      # partial states and their sum
    assert (out == 7.0).all() and words.tolist() == [0, 0, 0, 0]
    words[0] = -6
    la.linattn_state(k, v, out=out, workspace=ws)
    assert torch.equal(out, want) and la.workspace_status(ws) == -6


# launches of a step: state and apply when the CTAs of a unit are a cluster, the sum of partial states between them otherwise
@pytest.mark.parametrize("dtype,B,N,H,d,rope,launches", [
    ("f32", 2, 300, 3, 112, True, 2), ("f32", 1, 300, 20, 112, False, 2), ("f32", 2, 200, 80, 64, False, 2),
    ("bf16", 2, 700, 5, 72, True, 2), ("bf16", 2, 300, 80, 40, True, 2), ("f32", 2, 6000, 10, 112, True, 3),
    ("f32", 1, 6000, 20, 112, False, 3), ("bf16", 1, 6000, 40, 96, True, 3), ("f32", 2, 900, 100, 32, True, 2)])
def test_both_sums_of_a_unit(la, dtype, B, N, H, d, rope, launches):
    """A read-only step and two steps through the cache, by clusters and by partial states, several batch entries, more units than
    SMs.  Bars on the 2-norm as above: 2^-22 for S and z on top of fp16 tables taken as they are."""
    q, k, v = (to_dev(x) for x in gen(B, N, H, d, 7800 + N + d, dtype))
    table = tab = None
    if rope:
        cos, sin = synth.rope_table(1, 1, N, d)
        table = la.rope_pack(to_dev(cos), to_dev(sin))
        tab = table.cpu().numpy().astype(np.float64)
    qn, kn, vn = to_f64(q).clip(0), to_f64(k).clip(0), to_f64(v)
    S = (turned(kn, tab).transpose(0, 2, 3, 1) @ vn.transpose(0, 2, 1, 3)).swapaxes(-1, -2)
    z = kn.sum(1)
    cache = la.BlockLinCache(B, H, d, q.dtype, "cuda", max_T_b=N, eps=EPS)
    for steps in (1, 2):
        args = (q, k, v, table) if rope else (q, k, v)
        before = la.load_library().linattn_kernel_launches()
        peek = cache.peek_rope(*args) if rope else cache.peek(*args)
        assert la.load_library().linattn_kernel_launches() == before + launches
        o = cache.step_rope(*args) if rope else cache.step(*args)
        assert la.load_library().linattn_kernel_launches() == before + 2 * launches
        st = to_f64(cache.state)
        assert relative(st[:, :, :d], steps * S) <= 2.0 ** -22 and relative(st[:, :, d], steps * z) <= 2.0 ** -22
        O = turned(qn, tab).transpose(0, 2, 1, 3) @ (steps * S).swapaxes(-1, -2)
        O = (O / ((qn.transpose(0, 2, 1, 3) @ (steps * z)[..., None]) + EPS)).transpose(0, 2, 1, 3)
        assert relative(to_f64(o), O) <= (2.0 ** -21 if dtype == "f32" else 2.0 ** -9) and (o == peek).all()
    assert cache.status() == 0


@pytest.mark.parametrize("d,rope", [(24, False), (64, True), (112, False)])
@pytest.mark.parametrize("value", [3.4e38, 3e38, float("inf")])
def test_queries_that_the_denominator_does_not_see(la, d, rope, value):
    """Where no key has a feature (or neither of a pair), z and S are zero there: the largest finite queries count for nothing, an
    infinite one makes its row NaN.  The rows around it stay as they are."""
    import torch

    B, N, H = 1, 200, 2
    q, k, v = (to_dev(x) for x in gen(B, N, H, d, 7900 + d, "f32"))
    k[..., 4:6] = -1.0
    table = None
    if rope:
        cos, sin = synth.rope_table(1, 1, N, d)
        table = la.rope_pack(to_dev(cos), to_dev(sin))
    call = (lambda: la.linattn_forward_rope(q, k, v, table, EPS)) if rope else (lambda: la.linattn_forward(q, k, v, EPS))
    q[..., 4:6] = 0.0
    want = call()
    q[0, 100, 1, 4] = value
    got = call()
    if value == float("inf"):
        assert got[0, 100, 1].isnan().all()
        got[0, 100, 1] = want[0, 100, 1]
    assert relative(to_f64(got), to_f64(want)) <= 2.0 ** -21
