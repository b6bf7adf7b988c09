"""Small problems, where one CTA takes a whole unit: token counts around the 64-token stages, the 128-token tiles and the
line behind which the whole grid takes the work, every tensor-core head dim, head counts that leave a packed group partly
empty, all modes on one shape with the same bits.  (From 129 tokens on lone CTAs have the calls of too many units for clusters.)"""
import numpy as np
import pytest

import synth
from parity_util import assert_parity_bf16, assert_state_close, to_dev, to_f64

pytestmark = pytest.mark.gpu

EPS = 1e-6


@pytest.fixture(scope="module")
def la():
    import torch

    assert torch.cuda.is_available(), "these tests need a CUDA device"
    import paper_2509_24695_b200 as la

    la.load_library()
    return la


def gen(B, N, H, d, seed):
    return tuple(synth.gauss((B, N, H, d), seed, t) for t in (1, 2, 3))


@pytest.mark.parametrize("shape", [(1, 64, 3, 112), (2, 65, 2, 112), (1, 129, 3, 112), (1, 384, 2, 112), (1, 385, 2, 112),
                                   (1, 512, 50, 112), (1, 513, 50, 112), (1, 1, 2, 128), (2, 127, 3, 128), (1, 384, 2, 128),
                                   (1, 63, 3, 64), (2, 300, 5, 64), (1, 128, 5, 32), (2, 383, 6, 32), (1, 129, 149, 64), (2, 192, 150, 32),
                                   (1, 192, 101, 112)],
                         ids=lambda s: "B%d_N%d_H%d_d%d" % s)
def test_all_modes(la, orc, shape):
    import torch

    B, N, H, d = shape
    q, k, v = (to_dev(x) for x in gen(B, N, H, d, 8000 + N + d))
    qn, kn, vn = gen(B, N, H, d, 8000 + N + d)
    k0, v0 = gen(B, 40, H, d, 8100 + N + d)[1:]
    S, z = orc.state(kn, vn)
    S0, z0 = orc.state(k0, v0)
    st = la.linattn_state(k, v)
    assert_state_close(to_f64(st), S, z, 1e-5, "state")
    o = la.linattn_forward(q, k, v, EPS)
    assert_parity_bf16(to_f64(o), orc.forward(qn, kn, vn, EPS), "forward")
    assert torch.equal(o, la.linattn_apply(q, st, EPS))
    # a cache with a past: read-only, then committed, plain and with rotary factors
    cos, sin = synth.rope_table(1, 1, N + 40, d)
    table = la.rope_pack(to_dev(cos), to_dev(sin))
    packed = table.cpu().numpy().astype(np.float64)
    cat = [np.concatenate([a, b], axis=1) for a, b in ((gen(B, 40, H, d, 8100 + N + d)[0], qn), (k0, kn), (v0, vn))]
    for rope in (False, True):
        cache = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=max(N, 40), eps=EPS)
        if rope:
            cache.step_rope(None, to_dev(k0), to_dev(v0), table[:40].contiguous())
            args = (q, k, v, table[40:].contiguous())
            peek, step, ref = cache.peek_rope, cache.step_rope, orc.rope_forward(*cat, packed[..., 0], packed[..., 1], EPS)
        else:
            cache.step(None, to_dev(k0), to_dev(v0))
            args = (q, k, v)
            peek, step, ref = cache.peek, cache.step, orc.forward(*cat, EPS)
        before = cache.state.clone()
        o_peek = peek(*args)
        assert torch.equal(cache.state, before)
        o_step = step(*args)
        assert torch.equal(o_peek, o_step)
        # every block sees itself and its past: the second block's outputs are those of the whole sequence
        assert_parity_bf16(to_f64(o_step), ref[:, 40:], "step", rms_rel=1.5e-2 if rope else 1e-2)
        if not rope:
            assert_state_close(to_f64(cache.state), S + S0, z + z0, 1e-5, "cache")
        assert cache.status() == 0


@pytest.mark.parametrize("rope", [False, True])
@pytest.mark.parametrize("shape", [(1, 65, 3, 112), (1, 128, 2, 112), (1, 128, 2, 128), (1, 192, 3, 64), (2, 192, 6, 32), (1, 192, 101, 112),
                                   (1, 192, 150, 64), (1, 192, 296, 64), (2, 180, 151, 32)],
                         ids=lambda s: "B%d_N%d_H%d_d%d" % s)
def test_tiles_are_added_round_to_nearest(la, shape, rope):
    """The tensor core truncates when it adds into an accumulator.  Four steps of sixteen tokens leave 2^24 each; what the later
    tiles add to that, 1.5 a step, is below the last place of 2^24 and would be cut off there, but not of the sum of whole
    tiles: 2^26 and 6 a tile, of which a tile of one token has 1.5."""
    import torch

    B, N, H, d = shape
    v = torch.zeros(B, N, H, d, device="cuda")
    v[:, 0:64:16] = 2.0 ** 24
    v[:, 64::16] = 1.5
    q = k = torch.ones_like(v).bfloat16()
    v = v.bfloat16()
    want = np.float32(2.0 ** 26)
    for tile in range(64, N, 64):
        want = np.float32(want + np.float32(1.5 * len(range(tile, min(tile + 64, N), 16))))
    cache = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=N, eps=EPS)
    if rope:
        table = la.rope_pack(torch.ones(N, d // 2, device="cuda"), torch.zeros(N, d // 2, device="cuda"))
        cache.step_rope(q, k, v, table)
    else:
        cache.step(q, k, v)
        assert torch.equal(la.linattn_state(k, v), cache.state)
    assert (cache.state[:, :, :d] == float(want)).all() and (cache.state[:, :, d] == N).all()
    (cache.step_rope(None, k, v, table) if rope else cache.step(None, k, v))   # on top of an old state
    again = want
    for tile in range(0, N, 64):
        again = np.float32(again + (np.float32(2.0 ** 26) if tile == 0 else np.float32(1.5 * len(range(tile, min(tile + 64, N), 16)))))
    assert (cache.state[:, :, :d] == float(again)).all() and (cache.state[:, :, d] == 2 * N).all()


@pytest.mark.parametrize("N,units,d", [(129, 75, 64), (192, 148, 64), (129, 75, 32), (192, 148, 32), (192, 101, 112), (192, 148, 128), (128, 1, 112)])
@pytest.mark.parametrize("rope", [False, True])
def test_no_cluster_takes_these(la, N, units, d, rope):
    """What the shapes of many units are there for: that many clusters do not fit on the GPU at once."""
    assert la.cluster_ctas(1, units * {32: 4, 64: 2}.get(d, 1), d, N, rope) == 0


@pytest.mark.parametrize("shape", [(1, 63, 3, 64), (2, 128, 2, 112), (1, 129, 3, 112), (1, 192, 5, 64), (1, 193, 5, 64), (2, 191, 6, 32), (1, 128, 2, 128),
                                   (1, 192, 100, 112), (1, 192, 150, 64), (2, 130, 151, 32)], ids=lambda s: "B%d_N%d_H%d_d%d" % s)
def test_rotary_sums_in_the_cache(la, shape):
    """What rotary steps leave in the cache: z, of the plain keys, as exact as without rotary factors; S, of turned keys rounded
    to bf16 (2^-9 each, so 2^-9 of the sums' random part: its 2-norm)."""
    import torch

    B, N, H, d = shape
    q, k, v = gen(B, N, H, d, 8200 + N + d)
    cos, sin = synth.rope_table(1, 1, N, d)
    table = la.rope_pack(to_dev(cos), to_dev(sin))
    tab = table.cpu().numpy().astype(np.float64)
    cache = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=N, eps=EPS)
    kn, vn = to_f64(to_dev(k)).clip(0), to_f64(to_dev(v))
    c, s = tab[None, :, None, :, 0], tab[None, :, None, :, 1]
    a, b = kn[..., 0::2], kn[..., 1::2]
    S = np.einsum("bnhi,bnhj->bhji", np.stack((a * c - b * s, b * c + a * s), axis=-1).reshape(kn.shape), vn)
    z = kn.sum(1)
    for steps in (1, 2):
        cache.step_rope(to_dev(q) if steps == 2 else None, to_dev(k), to_dev(v), table)
        st = to_f64(cache.state)
        assert np.abs(st[:, :, d] - steps * z).max() <= 1e-6 * steps * z.max()
        err = np.sqrt(((st[:, :, :d] - steps * S) ** 2).sum() / ((steps * S) ** 2).sum())
        assert err <= 2.0 ** -9, err
