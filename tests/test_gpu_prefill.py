"""Prefill of several blocks in one launch against its three parts (every block's own state, their running sums on top of the cache, every
block's queries against its sum): the same bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

la = pytest.importorskip("paper_2509_24695_b200")


@pytest.mark.parametrize("B,M,T,H,d", [
    (1, 7, 4680, 20, 112),    # a column CTA and a few trailing tiles to a unit
    (1, 2, 7001, 3, 112),     # many columns to a unit, ragged last tile
    (2, 3, 2500, 25, 112),    # more units than CTAs
    (1, 16, 900, 40, 112),    # many units, operand images do not fit
    (3, 2, 1300, 18, 128),
    (1, 5, 3333, 35, 64),     # packed heads, the last group half full
    (2, 2, 5000, 6, 32),
    (1, 40, 321, 30, 64),
])
def test_prefill_is_its_parts(B, M, T, H, d):
    assert T > 192 and la.cluster_ctas(B * M, H, d, T) == 0   # the grid
    gen = torch.Generator(device="cuda").manual_seed(7 * T + M)
    q, k, v = (torch.randn(B, M * T, H, d, device="cuda", generator=gen).bfloat16() for _ in range(3))
    cache = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=T, prefill_blocks=M)
    cache.step(None, k[:, :T].contiguous(), v[:, T:2 * T].contiguous())
    run = cache.state.clone()
    before = la.kernel_launches()
    got = cache.prefill(q, k, v, M)
    assert la.kernel_launches() == before + 1
    assert cache.info()["blocks_seen"] == M + 1 and cache.info()["tokens_seen"] == (M + 1) * T

    split = [t.view(B * M, T, H, d) for t in (q, k, v)]
    own = la.linattn_state(split[1], split[2]).view(B, M, H, d + 1, d)
    states = []
    for m in range(M):
        run = run + own[:, m]
        states.append(run)
    want = la.linattn_apply(split[0], torch.stack(states, dim=1).view(B * M, H, d + 1, d).contiguous())
    assert torch.equal(cache.state, run)
    assert torch.equal(got.view(B * M, T, H, d), want)
    assert cache.status() == 0
