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


# Queries whose entries exceed the registers go through a path that reads them again in every pass.
@pytest.mark.parametrize("nlist,nq,nprobe,bf16", [
    (8192, 200, 96, True), (16_384, 300, 40, False), (16_384, 300, 64, False), (65_536, 100, 64, True), (65_536, 100, 96, True),
    (65_536, 100, 120, False), (16_384, 1000, 80, True), (8192, 40, 96, False), (65_536, 64, 100, True), (65_536, 64, 120, False),
    (131_072, 100, 104, True)])
def test_a_selections_registers_hold_the_entries_that_the_lists_leave(nlist, nq, nprobe, bf16):
    ix = _index(nlist, bf16=bf16)
    g = torch.Generator(device="cuda")
    g.manual_seed(nq)
    q = torch.randn(nq, 64, generator=g, device="cuda")
    plan = ix.rago_debug_search_plan(nq, nprobe, 1)
    assert plan["route"] == "lists" and plan["pilot_cols"] > 0
    ws = torch.zeros(ix.search_workspace_bytes(nq, nprobe, 1), dtype=torch.uint8, device="cuda")
    ix.rago_search_probes(q, nprobe, workspace=ws)
    torch.cuda.synchronize()
    ix.rago_check(ws)
    at = 256 * plan["counts_at"]
    items = ws[at:at + 4 * nq * plan["lists"]].view(torch.int32).view(nq, -1).sum(1)
    assert int(items.min()) >= nprobe + 8
    allowed = 0.02 if nq <= 888 else 0.25  # of the queries: the largest ones end a batch that fits the GPU at once
    assert float((items > plan["slots"]).float().mean()) <= allowed, (int(items.max()), plan["slots"])
    ix.close()


# Tiles of 480 (48 bytes), 256 (80) and 384 (96) vectors.  Few probes per list, many; lists of 47 000 vectors beyond L2, in it.
@pytest.mark.parametrize("N,nlist,M,nq,nprobe,prefetch", [
    (3_000_000, 64, 48, 600, 32, 1), (400_000, 64, 48, 600, 32, 0), (3_000_000, 512, 48, 600, 32, 0), (3_000_000, 512, 48, 60, 32, 1),
    (3_000_000, 64, 80, 40, 64, 1), (3_000_000, 64, 96, 40, 64, 0), (3_000_000, 64, 96, 4, 64, 1), (3_000_000, 64, 64, 1, 64, 0)])
def test_scan_prefetches_what_comes_from_dram(N, nlist, M, nq, nprobe, prefetch):
    ix = _index(nlist, d=2 * M, M=M, N=N, metric="ip")
    assert ix.rago_debug_search_plan(nq, nprobe, 10)["prefetch"] == prefetch
    ix.close()


# With 8192 lists the pilot pass ends behind nprobe = 120, with 65 536 candidate lists grow at 377 and end at 953.
@pytest.mark.parametrize("nlist,nq,nprobes", [(8192, 17, (8, 120, 121, 128, 400)), (8192, 300, (1, 64, 120, 121, 1024)),
                                              (65_536, 100, (16, 376, 377, 952, 953, 1016)), (255, 64, (1, 8, 255)),
                                              (20_001, 1500, (20, 376, 377, 953))])
def test_a_workspace_also_serves_fewer_probes(nlist, nq, nprobes):
    ix = _index(nlist)
    sizes = [ix.search_workspace_bytes(nq, p, 100) for p in nprobes]
    assert sizes == sorted(sizes)
    g = torch.Generator(device="cuda")
    g.manual_seed(nq)
    q = torch.randn(nq, 64, generator=g, device="cuda")
    ws = torch.zeros(sizes[-1], dtype=torch.uint8, device="cuda")
    for p in nprobes:
        ids, _ = ix.rago_search(q, p, 10, workspace=ws)  # refused if it asked for more than the largest nprobe did
        ix.rago_check(ws)
        assert int((ids >= 0).sum()) > 0
    ix.close()


# The start of a query weighs 7 us where the candidate buffer holds 4 096 keys, 17 where it holds 2 048, 5.5 for a small k, in tiles of 36 000
# bytes a us (at least 0.8 us each): buffers of 2 048 are those of 80 and 128 bytes.
@pytest.mark.parametrize("M,k,lead", [(48, 100, 5), (96, 100, 5), (64, 100, 4), (32, 100, 8), (80, 100, 21), (128, 100, 17), (48, 20, 4), (96, 20, 4)])
def test_the_weight_of_a_query_start_goes_by_the_candidate_buffer(M, k, lead):
    ix = _index(64, d=4 * M, M=M, N=200_000)
    assert ix.rago_debug_search_plan(400, 32, k)["lead"] == lead
    ix.close()


# Tiles of 46 KB (48 and 96 bytes) from one probe per list on; lists of 640 KB of 48-byte codes (13 654 vectors) however often they are probed.
@pytest.mark.parametrize("N,nlist,M,nq,nprobe,prefetch", [
    (400_000, 512, 96, 15, 32, 0), (400_000, 512, 96, 16, 32, 1), (400_000, 512, 96, 64, 32, 1), (400_000, 512, 96, 65, 32, 0),
    (400_000, 512, 48, 15, 32, 0), (400_000, 512, 48, 16, 32, 1), (400_000, 512, 128, 1, 32, 1), (400_000, 512, 32, 1, 32, 1),
    (3_004_000, 220, 48, 600, 32, 1), (3_003_000, 220, 48, 600, 32, 0), (2_800_000, 187, 48, 600, 32, 1), (2_700_000, 187, 48, 600, 32, 0)])
def test_scan_prefetches_by_the_bytes_of_tiles_and_lists(N, nlist, M, nq, nprobe, prefetch):
    ix = _index(nlist, d=2 * M, M=M, N=N, metric="ip")
    assert ix.rago_debug_search_plan(nq, nprobe, 10)["prefetch"] == prefetch
    ix.close()
