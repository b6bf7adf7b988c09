"""Rotary tensor-core path: where the rotations of a tile end.  The state pass fetches those of a 64-token stage in one copy, as
many as there are tokens; the apply pass loads them row by row.  What lies behind the table is NaN here and must not be seen."""
import numpy as np
import pytest

import synth
from parity_util import assert_parity_bf16, to_dev, to_f64

pytestmark = pytest.mark.gpu

EPS = 1e-6


@pytest.mark.parametrize("H,d", [(3, 112), (2, 128), (5, 64), (6, 32)])
@pytest.mark.parametrize("N", [1, 65, 449, 479, 480, 481, 511, 1537])
def test_nothing_behind_the_table_is_seen(orc, H, d, N):
    import torch

    import paper_2509_24695_b200 as la

    q, k, v = (synth.gauss((1, N, H, d), 8500 + N + d, t) for t in (1, 2, 3))
    cos, sin = synth.rope_table(1, 1, N, d)
    room = torch.full((N + 200, d // 2, 2), float("nan"), dtype=torch.float16, device="cuda")
    table = room[:N]
    table.copy_(la.rope_pack(to_dev(cos), to_dev(sin)))
    tab = table.cpu().numpy().astype(np.float64)
    o = la.linattn_forward_rope(to_dev(q), to_dev(k), to_dev(v), table, EPS)
    assert_parity_bf16(to_f64(o), orc.rope_forward(q, k, v, tab[..., 0], tab[..., 1], EPS), f"N={N} d={d}", rms_rel=1.5e-2)
    cache = la.BlockLinCache(1, H, d, torch.bfloat16, "cuda", max_T_b=N, eps=EPS)
    assert torch.equal(cache.step_rope(to_dev(q), to_dev(k), to_dev(v), table), o)
    z = to_f64(to_dev(k)).clip(0).sum(1)
    assert np.abs(to_f64(cache.state)[:, :, d] - z).max() <= 1e-6 * z.max() and torch.isfinite(cache.state).all()
