"""Kernels that may start early and use tensor memory: it is allocated behind the wait for the grids before, and before the next grid may
start.  Otherwise a CTA of a neighbouring grid on the same SM could hold what this one waits for, and wait for this one."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2509_24695_b200", "csrc")
KERNELS = [("umma_cluster.cuh", "umma_cluster_kernel"), ("umma_kernels.cu", "umma_fused_kernel"), ("split_kernels.cu", "split_state_kernel"),
           ("split_kernels.cu", "split_apply_kernel")]


@pytest.mark.parametrize("file,kernel", KERNELS)
def test_tensor_memory_between_wait_and_next(file, kernel):
    text = open(os.path.join(CSRC, file)).read()
    start = re.search(r"__global__[^{;]*?\b%s\(" % kernel, text, re.S).start()
    end = text.find("__global__", start + 10)
    body = text[start:end if end > 0 else len(text)]
    at = [[m.start() for m in re.finditer(call, body)] for call in (r"wait_for_prior_grids\(\);", r"tmem_alloc\(", r"let_next_grid_start\(\);")]
    assert [len(a) for a in at] == [1, 1, 1]
    assert at[0][0] < at[1][0] < body.index("__syncthreads();", at[1][0]) < at[2][0]
