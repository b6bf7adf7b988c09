"""Small problems, where one CTA takes a whole unit: token counts around the 64-token stages, the 128-token tiles and the
line behind which the whole grid takes the work, every tensor-core head dim, head counts that leave a packed group partly
empty, all modes on one shape with the same bits."""
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
                                   (1, 63, 3, 64), (2, 300, 5, 64), (1, 128, 5, 32), (2, 383, 6, 32)],
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
