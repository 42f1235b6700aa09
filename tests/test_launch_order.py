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


def test_the_scan_waits_before_it_reads_global_memory_or_exits():
    text = open(os.path.join(ROOT, "paper_2503_14649_b200", "csrc", "scan.cu")).read()
    body = text[text.index("scan_kernel(const ScanArgs a)"):]
    body = re.sub(r"//[^\n]*", "", body[:body.index("\n}\n")])
    # unconditional: statements of their own, the first in the exit of a plan that does not fit, the second in front of all else
    waits = [m.start() for m in re.finditer(r"[;{}]\s*grid_dependency_wait\(\);", body)]
    assert len(waits) == 2 and body.count("grid_dependency_wait") == 2
    assert body.index("if (!P.ok)") < waits[0] < body.index("return;") < waits[1]
    head = body[:waits[0]] + body[body.index("return;"):waits[1]]
    arguments = set(re.findall(r"\ba\.(\w+(?:\.\w+)?)", head))
    assert arguments <= {"stages", "dyn_bytes", "d", "vterm"} and "a.vterm != nullptr" in head, arguments  # no memory behind them
    assert waits[1] < body.index("grid_dependents_may_launch")
