"""Which batches are looked through for pairs of queries, and what larger batches and other kinds of calls with pairs answer."""

import pytest
import torch

from paper_2503_14649_b200 import binding

pytestmark = pytest.mark.gpu


def _even(M, N, nlist, seed=0):
    """Random codes in lists of (almost) equal length around random centroids."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed + M)
    c = torch.randn(nlist, 4 * M, generator=g, device="cuda")
    books = 0.3 * torch.randn(M, 256, 4, generator=g, device="cuda")
    codes = torch.randint(0, 256, (N, M), generator=g, device="cuda", dtype=torch.uint8)
    offsets = (torch.arange(nlist + 1, device="cuda", dtype=torch.int64) * N) // nlist
    return binding.rago_index_load(c, books, codes, offsets, torch.arange(N, device="cuda"), "l2"), c


def _launches(ix, q, nprobe, k):
    n = binding.rago_kernel_launches()
    ix.rago_search(q, nprobe, k)
    torch.cuda.synchronize()
    ix.rago_check()
    return binding.rago_kernel_launches() - n


# Pairs are looked for where sharing look-ups saves more than preparing and closing the pairs costs.  Not so: many queries over few
# vectors each (every pair is closed on a CTA), every list of a query matched with its partner's for little work.
@pytest.mark.parametrize("M,N,nlist,nq,nprobe,pairs", [
    (64, 2_200_000, 1024, 4000, 4, False), (96, 2_200_000, 1024, 4000, 8, False), (48, 2_200_000, 1024, 4000, 8, False),
    (48, 100_000, 1024, 1000, 1024, False), (48, 400_000, 1024, 1000, 1024, False),
    (96, 1_000_000, 512, 500, 256, True), (96, 2_000_000, 256, 300, 64, True), (16, 4_000_000, 256, 1000, 200, True)])
def test_pairs_are_looked_for_where_they_pay(M, N, nlist, nq, nprobe, pairs):
    ix, c = _even(M, N, nlist)
    g = torch.Generator(device="cuda")
    g.manual_seed(nq)
    q = (c[torch.randint(0, nlist, (nq,), generator=g, device="cuda")] + 0.3 * torch.randn(nq, 4 * M, generator=g, device="cuda")).contiguous()
    # k = 1024 is above the pairs' limit: the same launches without them
    assert _launches(ix, q, nprobe, 100) == _launches(ix, q, nprobe, 1024) + (5 if pairs else 0)
    ix.close()


# Pairs of 96-byte codes have a kernel of fewer warps for larger k: the values on both sides of the line, and the largest.
@pytest.mark.parametrize("k", [303, 304, 305, 448, 449, 512])
def test_pairs_of_96_byte_codes_for_larger_k_answer_as_single_queries_do(k):
    ix, c = _even(96, 400_000, 40)
    g = torch.Generator(device="cuda")
    g.manual_seed(k)
    q = (c[torch.arange(180, device="cuda") % 7] + 0.3 * torch.randn(180, 384, generator=g, device="cuda")).contiguous()
    assert _launches(ix, q, 24, k) == _launches(ix, q, 24, 1024) + 5
    ids, dists = ix.rago_search(q, 24, k)
    for b in range(0, 180, 60):  # batches that are too small for pairs
        i, s = ix.rago_search(q[b:b + 60].contiguous(), 24, k)
        assert torch.equal(ids[b:b + 60], i) and torch.equal(dists[b:b + 60].view(torch.int32), s.view(torch.int32)), b
    ix.close()


# Room for pairs is not a condition of a search: a workspace that lacks a little of it, or all of the pairs' tables, is searched one
# query at a time.
@pytest.mark.parametrize("M,k", [(64, 100), (96, 1), (16, 512)])
def test_a_workspace_without_room_for_pairs_is_searched_one_query_at_a_time(M, k):
    N, nlist, nq, nprobe = 64_000_000 // M, 4, 140, 3
    ix, c = _even(M, N, nlist)
    g = torch.Generator(device="cuda")
    g.manual_seed(k)
    q = (c[torch.arange(nq, device="cuda") % nlist] + 0.3 * torch.randn(nq, 4 * M, generator=g, device="cuda")).contiguous()
    need, staging = ix.search_workspace_bytes(nq, nprobe, k), ix.host_staging_bytes(nq, k)
    ids, dists = ix.rago_search(q, nprobe, k)
    alone = _launches(ix, q, nprobe, 1024)
    assert _launches(ix, q, nprobe, k) == alone + 5
    per_pair = {16: 32768, 64: 65536, 96: 98304}[M]  # the pair's table, in the part that may be missing
    for size, launches in ((need, alone + 5), (need - 256, alone), (need - nq // 2 * per_pair, alone)):
        ws = torch.empty(size + staging, dtype=torch.uint8, device="cuda")
        n = binding.rago_kernel_launches()
        i, s = ix.rago_search(q, nprobe, k, workspace=ws[:size])
        assert binding.rago_kernel_launches() - n == launches
        torch.cuda.synchronize()
        ix.rago_check(ws)
        assert torch.equal(i, ids) and torch.equal(s.view(torch.int32), dists.view(torch.int32))
        hi, hs = torch.empty((nq, k), dtype=torch.int64), torch.empty((nq, k))
        n = binding.rago_kernel_launches()
        ix.rago_search_host(q.cpu(), nprobe, k, hi, hs, ws)
        assert binding.rago_kernel_launches() - n == launches
        assert torch.equal(hi, ids.cpu()) and torch.equal(hs, dists.cpu())
        lists, _ = ix.rago_search_probes(q, nprobe, workspace=ws[:size])
        assert torch.equal(lists, ix.rago_search_probes(q, nprobe)[0])
    with pytest.raises(RuntimeError):
        ix.rago_search(q, nprobe, k, workspace=torch.empty(nq * per_pair, dtype=torch.uint8, device="cuda"))  # the tables of the queries alone
    ix.close()
