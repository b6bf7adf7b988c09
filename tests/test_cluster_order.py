"""The CTAs of a cluster go at their own pace, and a committing step writes the new sums of phi(k) where the old ones are: no CTA
may read the old ones when another may already have written."""
import os
import re

import numpy as np
import pytest

import synth
from parity_util import to_dev

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc")
EPS = 1e-6


def test_old_sums_are_read_by_the_thread_that_writes_them():
    """Reads and writes of the z row carry the same condition, which holds in one CTA of a cluster, and what is read goes into what
    that thread sends: it has been read before the others' sums, behind which the thread writes, can be complete."""
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, "umma_cluster.cuh")).read())
    statements = [" ".join(s.split()) for s in re.split(r"[;{}]", text)]
    owned = [s for s in statements if re.search(r"\bbool z_owned\b", s)]
    assert len(owned) == 1 and "rank == 0" in owned[0]
    reads = [s for s in statements if "p.state_base" in s and "z_at" in s]
    writes = [s for s in statements if "p.state[z_at" in s]
    assert len(reads) == 1 and reads[0].startswith("const float z_old = z_owned && p.accumulate ?")
    assert len(writes) == 1 and writes[0].startswith("if (z_owned && p.write_state)")
    sent = [i for i, s in enumerate(statements) if "store_async(" in s]
    assert len(sent) == 1 and statements.index(reads[0]) < sent[0] < statements.index(writes[0])
    assert any(s.startswith("const float z = z_old +") for s in statements[:sent[0]])


@pytest.mark.gpu
@pytest.mark.parametrize("rope,shape", [(True, (1, 1200, 4, 112)), (True, (1, 4680, 20, 112)), (True, (1, 700, 9, 64)), (True, (2, 200, 6, 32)),
                                        (True, (1, 500, 18, 128)), (False, (1, 700, 9, 64)), (False, (2, 200, 6, 32)), (False, (1, 192, 18, 128))],
                         ids=str)
def test_many_commits_see_what_the_read_only_step_saw(rope, shape):
    import torch

    import paper_2509_24695_b200 as la

    B, N, H, d = shape
    q, k, v, k0, v0 = (to_dev(synth.gauss(shape, 8700 + N + d, t)) for t in range(1, 6))
    table = la.rope_pack(*(to_dev(t) for t in synth.rope_table(1, 1, N, d)))
    cache = la.BlockLinCache(B, H, d, torch.bfloat16, "cuda", max_T_b=N, eps=EPS)
    past = (lambda: cache.step_rope(None, k0, v0, table)) if rope else (lambda: cache.step(None, k0, v0))
    args = (q, k, v, table) if rope else (q, k, v)
    peek, step = (cache.peek_rope, cache.step_rope) if rope else (cache.peek, cache.step)
    past()
    old = cache.state.clone()
    seen = peek(*args)
    step(*args)
    new = cache.state.clone()
    differ = torch.zeros((), dtype=torch.int64, device="cuda")
    for _ in range(300):
        cache.state.copy_(old)
        differ += (step(*args) != seen).sum() + (cache.state != new).sum()
    assert differ.item() == 0 and cache.status() == 0
    z = k.float().clamp_min(0).double().sum(1) + k0.float().clamp_min(0).double().sum(1)
    assert np.abs((new[:, :, d].double() - z).cpu().numpy()).max() <= 1e-6 * z.max().item()


def test_old_state_is_asked_for_before_queries_are_clamped():
    """The loads of the old state are on their way while the clamping goes on, and are used behind the sums' arrival."""
    body = open(os.path.join(CSRC, "umma_cluster.cuh")).read()
    asked = [m.start() for m in re.finditer(r"= __ldcg\(reinterpret_cast<const float4\*>\(base", body)]
    clamped, used = body.index("mbar_test(x_full"), body.index("mbar_wait_cluster(x_full")
    assert asked and max(asked) < clamped < used
