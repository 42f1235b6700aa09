"""The rules that choose a search's kernels by its sizes: which side of each rule a call falls on, through
rago_debug_search_plan, where the other side was measured to be the slower one."""

import pytest
import torch

from paper_2503_14649_b200 import binding

pytestmark = pytest.mark.gpu


def _index(nlist, d=64, M=16, N=2000, metric="l2", bf16=False, seed=0):
    """Random centroids, codebooks and codes; lists of (almost) equal length."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + nlist)
    c = torch.randn(nlist, d, generator=g, device="cuda")
    books = torch.randn(M, 256, d // M, generator=g, device="cuda")
    codes = torch.randint(0, 256, (N, M), generator=g, device="cuda", dtype=torch.uint8)
    offsets = (torch.arange(nlist + 1, device="cuda") * N) // nlist
    return binding.rago_index_load(c.bfloat16() if bf16 else c, books, codes, offsets, torch.arange(N, device="cuda"), metric)


@pytest.mark.parametrize("nlist,nq,early", [(300, 64, 1), (4096, 64, 1), (18_001, 17, 1), (19_200, 17, 0), (65_536, 100, 0), (8192, 500, 0)])
def test_only_a_launch_that_leaves_sms_idle_lets_its_successor_start(nlist, nq, early):
    ix = _index(nlist)
    assert ix.rago_debug_search_plan(nq, 32, 10)["early_successor"] == early
    ix.close()


# The sample is every 16th list of at least 8192 and holds four times the wanted lists; lists hold at most 960 wanted ones.
@pytest.mark.parametrize("nlist,nprobe,cols", [(8192, 120, 512), (8192, 121, 0), (8176, 8, 0), (8193, 8, 0), (65_536, 952, 4096), (65_536, 953, 0)])
def test_pilot_pass(nlist, nprobe, cols):
    ix = _index(nlist)
    assert ix.rago_debug_search_plan(100, nprobe, 10)["pilot_cols"] == cols
    ix.close()
