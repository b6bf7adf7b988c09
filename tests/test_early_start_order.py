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


def body_of(file, kernel):
    text = re.sub(r"//[^\n]*", "", open(os.path.join(CSRC, file)).read())
    start = re.search(r"__global__[^{;]*?\b%s\(" % kernel, text, re.S).start()
    end = text.find("__global__", start + 10)
    return text[start:end if end > 0 else len(text)]


GRID_ONLY = {"zrow"}   # read by the cooperative form of umma_fused_kernel alone, which does not start early


@pytest.mark.parametrize("file,kernel", KERNELS + [("tconv.cu", "tconv_kernel"), ("tconv.cu", "tconv_step_kernel")])
def test_loads_that_may_move_have_their_pointer_from_behind_the_wait(file, kernel):
    body = body_of(file, kernel)
    loads = re.findall(r"__ld(?:g|cg|cs|ca|lu)\(\s*(?:reinterpret_cast<[^()]*>\()?\s*(?:static_cast<[^()]*>\()?\s*([\w.>-]+)", body)
    assert len(loads) == len(re.findall(r"__ld(?:g|cg|cs|ca|lu)\(", body)) and (loads or kernel == "split_state_kernel")

    def behind(name):   # every value that the name has in this kernel
        made = re.findall(r"(?<![\w.>])%s = ([^;]*);" % re.escape(name), body)
        return bool(made) and all("behind_wait(" in m or behind(re.search(r"static_cast<[^()]*>\((\w+)\)|(\w+)", m).group(1) or "") for m in made)

    for name in set(loads) - GRID_ONLY - {"behind_wait"}:
        assert behind(name), name
