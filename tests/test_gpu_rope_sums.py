"""Sums of rotary steps on clusters: the tensor core truncates when it adds into an accumulator, so it matters how many additions one
takes.  Factors that turn nothing leave the keys as they are; then the sums are as exact as without rotary factors."""
import numpy as np
import pytest

import synth
from parity_util import to_dev, to_f64

pytestmark = pytest.mark.gpu

EPS = 1e-6


def states(N, H, d, seed):
    import torch

    import paper_2509_24695_b200 as la

    k, v = (synth.gauss((1, N, H, d), seed, t) for t in (2, 3))
    table = la.rope_pack(torch.ones(N, d // 2, device="cuda"), torch.zeros(N, d // 2, device="cuda"))
    cache = la.BlockLinCache(1, H, d, torch.bfloat16, "cuda", max_T_b=N, eps=EPS)
    cache.step_rope(None, to_dev(k), to_dev(v), table)
    assert cache.status() == 0
    return cache.state[:, :, :d], la.linattn_state(to_dev(k), to_dev(v))[:, :, :d], k, v


@pytest.mark.parametrize("N,H,d", [(129, 3, 64), (192, 3, 64), (192, 35, 64), (300, 4, 112), (512, 5, 112), (150, 6, 32), (190, 3, 128)])
def test_one_tile_a_cta(N, H, d):
    """Four steps of sixteen tokens, an accumulator for each, added up round to nearest: the same bits with and without factors."""
    import torch

    turned, plain, _, _ = states(N, H, d, 8800 + N + d)
    assert torch.equal(turned, plain)


@pytest.mark.parametrize("N,H,d", [(1200, 4, 112), (4680, 20, 112), (1536, 4, 64), (900, 18, 128)])
def test_several_tiles_a_cta(N, H, d):
    """A chain as long as the CTA has tiles, n: each addition cuts off less than 2^-23 of the accumulator's partial sum, which is at most
    the whole sum of magnitudes, on average half of that, and so do the additions of the owner, rounded: n 2^-23 of the magnitudes."""
    turned, _, k, v = states(N, H, d, 8800 + N + d)
    kn, vn = to_f64(to_dev(k))[0].clip(0).transpose(1, 2, 0), to_f64(to_dev(v))[0].transpose(1, 0, 2)
    S, size = (kn @ vn).transpose(0, 2, 1), (kn @ np.abs(vn)).transpose(0, 2, 1)
    n = -(-(-(-N // 64)) // 2)
    assert (np.abs(to_f64(turned)[0] - S) <= min(n, 13) * 2.0 ** -23 * size).all()
