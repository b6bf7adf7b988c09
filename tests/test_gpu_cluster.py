"""Blocks whose units are taken by thread-block clusters: token counts that split evenly and unevenly over the CTAs, CTAs of
one 64-token tile and of several (an odd number leaves half an apply tile; enough of them that stages, accumulators and slots come
round again), clusters of two to eight, head counts that leave a packed group partly empty, all modes on one shape with the same
bits; and shapes just behind the line, which the grid takes."""
import numpy as np
import pytest

import synth
from parity_util import assert_parity_bf16, assert_state_close, to_dev, to_f64

pytestmark = pytest.mark.gpu

EPS = 1e-6
BOTH = [(1, 193, 3, 112), (1, 577, 2, 112), (2, 700, 10, 112), (2, 130, 37, 112), (1, 600, 26, 112), (1, 500, 33, 112), (1, 2000, 40, 112),
        (1, 1150, 45, 112), (1, 1536, 60, 112), (1, 150, 18, 128), (2, 192, 22, 128), (2, 333, 5, 64), (1, 2000, 80, 64), (1, 257, 6, 32), (2, 900, 70, 32)]
ROPE_ALONE = [(1, 1025, 5, 112), (1, 2100, 33, 112), (1, 260, 3, 128), (1, 1500, 18, 128), (1, 2000, 35, 64)]   # plain: the grid
CASES = [(rope, shape, True) for shape in BOTH for rope in (False, True)]
CASES += [(rope, shape, rope) for shape in ROPE_ALONE for rope in (False, True)] + [(True, (1, 5000, 7, 112), False), (True, (1, 2500, 34, 112), False)]


@pytest.fixture(scope="module")
def la():
    import torch

    assert torch.cuda.is_available(), "these tests need a CUDA device"
    import paper_2509_24695_b200 as la

    la.load_library()
    return la


def gen(B, N, H, d, seed):
    return tuple(synth.gauss((B, N, H, d), seed, t) for t in (1, 2, 3))


@pytest.mark.parametrize("rope,shape,clusters", CASES, ids=["%sB%d_N%d_H%d_d%d" % ("rope_" if c[0] else "", *c[1]) for c in CASES])
def test_all_modes(la, orc, shape, rope, clusters):
    import torch

    B, N, H, d = shape
    assert (la.cluster_ctas(B, H, d, N, rope) >= 2) == clusters
    qn, kn, vn = gen(B, N, H, d, 8300 + N + d)
    q, k, v = (to_dev(x) for x in (qn, kn, vn))
    k0, v0 = gen(B, 40, H, d, 8400 + N + d)[1:]
    cos, sin = synth.rope_table(1, 1, N + 40, d)
    table = la.rope_pack(to_dev(cos), to_dev(sin))
    tab = table.cpu().numpy().astype(np.float64)
    cat = [np.concatenate([a, b], axis=1) for a, b in ((qn[:, :1].repeat(40, axis=1), qn), (k0, kn), (v0, vn))]
    cache = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=max(N, 40), eps=EPS)
    S, z = orc.state(kn, vn)
    S0, z0 = orc.state(k0, v0)
    if rope:
        cache.step_rope(None, to_dev(k0), to_dev(v0), table[:40].contiguous())
        args, peek, step = (q, k, v, table[40:].contiguous()), cache.peek_rope, cache.step_rope
        ref = orc.rope_forward(*cat, tab[..., 0], tab[..., 1], EPS)[:, 40:]
        head = table[:N].contiguous()
        o = la.linattn_forward_rope(q, k, v, head, EPS)
        assert_parity_bf16(to_f64(o), orc.rope_forward(qn, kn, vn, tab[:N, :, 0], tab[:N, :, 1], EPS), "forward", rms_rel=1.5e-2)
        assert torch.equal(o, la.linattn_forward_rope(q, k, v, head, EPS))
    else:
        cache.step(None, to_dev(k0), to_dev(v0))
        args, peek, step, ref = (q, k, v), cache.peek, cache.step, orc.forward(*cat, EPS)[:, 40:]
        st = la.linattn_state(k, v)
        assert_state_close(to_f64(st), S, z, 1e-5, "state")
        o = la.linattn_forward(q, k, v, EPS)
        assert_parity_bf16(to_f64(o), orc.forward(qn, kn, vn, EPS), "forward")
        assert torch.equal(o, la.linattn_apply(q, st, EPS)) and torch.equal(st, la.linattn_state(k, v))
    before = cache.state.clone()
    o_peek = peek(*args)
    assert torch.equal(cache.state, before)
    o_step = step(*args)
    assert torch.equal(o_peek, o_step) and cache.status() == 0
    # every block sees itself and its past: the second block's outputs are those of the whole sequence
    assert_parity_bf16(to_f64(o_step), ref, "step", rms_rel=1.5e-2 if rope else 1e-2)
    zc = to_f64(cache.state)[:, :, d]
    assert np.abs(zc - (z + z0)).max() <= 1e-5 * (z + z0).max()
    if not rope:
        assert_state_close(to_f64(cache.state), S + S0, z + z0, 1e-5, "cache")
