"""A workspace made for a tensor holds what calls on it need, whatever its strides."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

la = pytest.importorskip("paper_2509_24695_b200")


@pytest.mark.parametrize("B,N,H,d", [(1, 8000, 70, 32), (3, 3000, 70, 32), (1, 8000, 20, 64), (1, 300, 4, 32)])
@pytest.mark.parametrize("rope", [False, True])
def test_head_major(B, N, H, d, rope):
    gen = torch.Generator(device="cuda").manual_seed(N)
    q, k, v = (torch.randn(B, H, N, d, device="cuda", generator=gen).bfloat16().permute(0, 2, 1, 3) for _ in range(3))
    ang = torch.rand(N, d // 2, device="cuda", generator=gen)
    tab = la.rope_pack(ang.cos(), ang.sin())

    def forward(*t):
        return la.linattn_forward_rope(*t, tab, workspace=la.new_rope_workspace(t[0])) if rope else la.linattn_forward(*t)

    got, want = forward(q, k, v), forward(*(t.contiguous() for t in (q, k, v)))
    assert got.stride() == q.stride()
    # other kernels for heads of 32: both round the output to bf16 (2^-9), and one of them the turned features too
    assert (got.float() - want.float()).norm() <= (2 ** -7 if rope else 2 ** -8) * want.float().norm()


def test_strides_that_no_call_takes():
    """Asked for all the same, for what the tensor will be copied to."""
    q = torch.zeros(2, 64, 500, 3, device="cuda", dtype=torch.bfloat16).permute(0, 2, 3, 1)
    assert la.new_workspace(q).numel() == la.new_workspace(q.contiguous()).numel()
    assert la.new_rope_workspace(q).numel() == la.new_rope_workspace(q.contiguous()).numel()
