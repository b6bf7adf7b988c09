"""fp32 apply pass whose MMAs take two parts of the queries at once (d > 96): token counts around its 64-token tiles, several tiles
to a CTA, against 64 bits.  Bar on the 2-norm: about 112 products and a quotient, 2^-21, as for one tile."""
import numpy as np
import pytest

import synth
from parity_util import to_dev, to_f64

pytestmark = pytest.mark.gpu

EPS = 1e-6


@pytest.mark.parametrize("d", [96, 100, 112, 116, 128])
@pytest.mark.parametrize("N", [1, 63, 64, 65, 127, 129, 193, 9000])
def test_outputs(d, N):
    import paper_2509_24695_b200 as la

    H = 20 if N > 1000 else 3
    q, k, v = (synth.gauss((1, N, H, d), 8600 + N + d, t, dtype="f32") for t in (1, 2, 3))
    st = la.linattn_state(to_dev(k), to_dev(v))
    W = to_f64(st)[0]
    qn = q[0].astype(np.float64).clip(0).transpose(1, 0, 2)
    ref = qn @ W[:, :d].transpose(0, 2, 1) / (qn @ W[:, d, :, None] + EPS)
    o = to_f64(la.linattn_apply(to_dev(q), st, EPS))[0].transpose(1, 0, 2)
    assert np.sqrt(((o - ref) ** 2).sum() / (ref ** 2).sum()) <= 2.0 ** -21
