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
    assert T > 192 and la.cluster_ctas(B * M, H, d, T) == 0   # the parts' state comes from the grid too: the same order
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


@pytest.mark.parametrize("B,M,T,H,d,launches", [
    (1, 7, 64, 20, 112, 3),     # blocks that lone CTAs take
    (1, 3, 130, 1, 32, 3),
    (2, 5, 700, 4, 112, 3),     # ... and clusters
    (1, 2, 33, 3, 128, 3),
    (1, 9, 1, 2, 64, 3),        # blocks of one token
    (1, 7, 600, 1, 112, 3),     # 70 records to a piece
    (1, 7, 1500, 2, 64, 3),
    (1, 7, 300, 20, 112, 1),    # blocks that the grid takes
    (1, 7, 257, 70, 32, 1),
])
def test_prefill_of_small_blocks(B, M, T, H, d, launches):
    """Against the steps, block by block: other forms, so to rounding (both sums of S within 1e-6 of 64 bits, outputs bf16)."""
    gen = torch.Generator(device="cuda").manual_seed(T + M)
    q, k, v = (torch.randn(B, M * T, H, d, device="cuda", generator=gen).bfloat16() for _ in range(3))
    one = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=T, prefill_blocks=M)
    steps = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=T)
    before = la.kernel_launches()
    got = one.prefill(q, k, v, M)
    assert la.kernel_launches() == before + launches
    cut = lambda t, m: t[:, m * T:(m + 1) * T].contiguous()
    want = torch.cat([steps.step(cut(q, m), cut(k, m), cut(v, m)) for m in range(M)], dim=1)
    assert (one.state - steps.state).norm() <= 2e-6 * steps.state.norm()
    # the same bf16 value, or a neighbour of it where the sums fall on both sides of the middle
    assert (got.float() - want.float()).abs().max() <= 2 ** -7 * want.float().abs().max()
    assert (got.float() - want.float()).norm() <= 1e-3 * want.float().norm()
    assert one.status() == 0


@pytest.mark.parametrize("B,M,T,H,d", [(1, 7, 64, 20, 112), (1, 7, 128, 70, 32), (2, 3, 132, 20, 112), (1, 2, 192, 35, 64), (1, 3, 107, 6, 128),   # lone CTAs
                                       (2, 5, 700, 4, 112), (1, 2, 2304, 20, 112), (1, 4, 900, 35, 64), (2, 7, 709, 9, 32),                    # clusters
                                       (1, 7, 300, 20, 112), (1, 3, 1500, 18, 128)])                                                        # the grid
def test_state_is_the_blocks_own(B, M, T, H, d):
    """Whatever takes a block's state in the other calls on its shape takes it here: with queries and without the cache is what the states of
    the blocks add up to, bit for bit, and as near to 64 bits."""
    gen = torch.Generator(device="cuda").manual_seed(T + d)
    q, k, v = (torch.randn(B, M * T, H, d, device="cuda", generator=gen).bfloat16() for _ in range(3))
    own = la.linattn_state(k.view(B * M, T, H, d), v.view(B * M, T, H, d)).view(B, M, H, d + 1, d)
    want = torch.zeros_like(own[:, 0])
    for m in range(M):
        want = want + own[:, m]
    for queries in (q, None):
        cache = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=T, prefill_blocks=M)
        cache.reset()
        cache.prefill(queries, k, v, M)
        assert torch.equal(cache.state, want)
