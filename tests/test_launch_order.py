"""Order of the steps at the head of the tensor-core kernel, read from its source (a run that got it wrong would stop the GPU)."""

import os
import re

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tensor_memory_is_taken_after_the_wait_for_the_kernel_in_front():
    text = open(os.path.join(ROOT, "paper_2503_14649_b200", "csrc", "gemm_select.cu")).read()
    body = text[text.index("gemm_select_kernel(const __grid_constant__"):]
    body = re.sub(r"//[^\n]*", "", body[:body.index("\n}\n")])
    wait, alloc = body.index("grid_dependency_wait();"), body.index("tmem_alloc_pair(")
    use = body.index("tmem_base = *tmem_slot")
    assert wait < alloc < body.index("cluster_sync_all();") < use
    assert body.index("fence_barrier_init();") < body.index("cluster_sync_all();")
