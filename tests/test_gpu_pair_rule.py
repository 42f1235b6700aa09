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


def _check_against_small_batches(ix, q, nprobe, k, size=64):
    ids, dists = ix.rago_search(q, nprobe, k)
    for b in range(0, q.shape[0], size):
        i, s = ix.rago_search(q[b:b + size].contiguous(), nprobe, k)
        assert torch.equal(ids[b:b + size], i) and torch.equal(dists[b:b + size].view(torch.int32), s.view(torch.int32)), b
    return ids, dists


def _uneven(M, dsub, sizes, metric, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    c = torch.randn(len(sizes), M * dsub, generator=g, device="cuda")
    books = 0.3 * torch.randn(M, 256, dsub, generator=g, device="cuda")
    N = sum(sizes)
    codes = torch.randint(0, 256, (N, M), generator=g, device="cuda", dtype=torch.uint8)
    offsets = torch.tensor([0] + sizes, device="cuda").cumsum(0)
    return binding.rago_index_load(c, books, codes, offsets, torch.randperm(N, generator=g, device="cuda"), metric), c


def _near(c, owners, seed=3):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (c[owners] + 0.3 * torch.randn(len(owners), c.shape[1], generator=g, device="cuda")).contiguous()


# Every warp of the ranking takes a second query from 1 185 on; 4 096 is the most, and fills the keys' array and the query's 12 bits.
# One more goes without pairs (and with tables that the scan builds, whose scale is another: its bits are not those of small batches).
@pytest.mark.parametrize("nq", [1185, 1300, 4095, 4096, 4097])
def test_batches_up_to_the_largest_with_pairs(nq):
    ix, c = _uneven(32, 4, [150_000, 100_000, 60_000] + [500 + i for i in range(50)], "l2", seed=nq)
    q = _near(c, torch.arange(nq, device="cuda") % 3 + 5 * (torch.arange(nq, device="cuda") % 101 == 0))
    assert _launches(ix, q, 5, 20) == _launches(ix, q, 5, 1024) + (5 if nq <= 4096 else 0)
    if nq <= 4096:
        _check_against_small_batches(ix, q, 5, 20)
    ix.close()


# Sub-spaces of 12 dimensions, many probes (entries of more than two rounds of 32 a list, with few and many lists that are not shared).
@pytest.mark.parametrize("M,dsub,metric,nq,nprobe,k", [(64, 12, "l2", 150, 10, 100), (32, 12, "ip", 200, 70, 10), (96, 4, "l2", 140, 129, 64),
                                                       (48, 4, "ip", 131, 200, 100)])
def test_pairs_with_twelve_dimensions_and_many_probes(M, dsub, metric, nq, nprobe, k):
    big = 450_000_000 // (M * nq)
    sizes = [7 * big + 1, 4 * big] + [300 + 7 * i for i in range(210)]
    ix, c = _uneven(M, dsub, sizes, metric, seed=M + dsub)
    q = _near(c, torch.tensor([0] * (nq // 2 | 1) + [1] * (nq // 4) + [3 * i % 212 for i in range(nq)], device="cuda")[:nq])
    assert _launches(ix, q, nprobe, k) == _launches(ix, q, nprobe, 1024) + 5
    _check_against_small_batches(ix, q, nprobe, k)
    ix.close()


def test_pairs_behind_the_two_level_quantiser_from_host_buffers_and_on_a_second_stream():
    sizes = [400_000, 250_000] + [1000 + i for i in range(62)]
    ix, c = _uneven(64, 4, sizes, "l2", seed=9)
    level1, children = c[:8].contiguous(), torch.arange(0, 65, 8, device="cuda", dtype=torch.int32)
    nq, nprobe, k = 150, 6, 50
    q = _near(c, torch.arange(nq, device="cuda") % 2)
    ids, dists = _check_against_small_batches(ix, q, nprobe, k)
    assert _launches(ix, q, nprobe, k) == _launches(ix, q, nprobe, 1024) + 5
    hi, hs = torch.empty((nq, k), dtype=torch.int64), torch.empty((nq, k))
    ws = torch.empty(ix.search_workspace_bytes(nq, nprobe, k) + ix.host_staging_bytes(nq, k), dtype=torch.uint8, device="cuda")
    ix.rago_search_host(q.cpu(), nprobe, k, hi, hs, ws)
    assert torch.equal(hi, ids.cpu()) and torch.equal(hs, dists.cpu())
    # two streams at once, each with its own workspace and its own queries
    other = _near(c, torch.arange(nq, device="cuda") % 2, seed=4)
    expected = [(ids, dists), tuple(t.clone() for t in ix.rago_search(other, nprobe, k))]
    torch.cuda.synchronize()
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    spaces = [torch.empty(ix.search_workspace_bytes(nq, nprobe, k), dtype=torch.uint8, device="cuda") for _ in streams]
    got = []
    for _ in range(5):
        for queries, stream, space in zip((q, other), streams, spaces):
            with torch.cuda.stream(stream):
                got.append(ix.rago_search(queries, nprobe, k, workspace=space))
    torch.cuda.synchronize()
    for n, (i, s) in enumerate(got):
        assert torch.equal(i, expected[n % 2][0]) and torch.equal(s, expected[n % 2][1])
    # the level above the centroids in front of the same scan (b1 = all nodes: every list is a candidate)
    ix.rago_index_set_coarse_tree(level1, children, 8)
    assert _launches(ix, q, nprobe, k) == _launches(ix, q, nprobe, 1024) + 5
    _check_against_small_batches(ix, q, nprobe, k)
    ix.close()


# Queries whose tables are not bounded have no partner, and no other query's answer changes: all of them compared, each in a batch too small for pairs.
def test_pairs_beside_queries_with_infinite_and_huge_values():
    ix, c = _uneven(64, 4, [900_000, 5000, 4000, 300], "l2", seed=5)
    q = _near(c, torch.tensor([0] * 80 + [1] * 17, device="cuda"))
    special = (3, 10, 11, 40)
    q[3, 5], q[10], q[11, 0] = float("inf"), float("nan"), 3e38
    q[40] *= 1e30
    assert _launches(ix, q, 3, 50) == _launches(ix, q, 3, 1024) + 5
    ids, dists = ix.rago_search(q, 3, 50)
    good = [i for i in range(97) if i not in special]
    for b in range(0, len(good), 60):
        i, s = ix.rago_search(q[good[b:b + 60]].contiguous(), 3, 50)
        assert torch.equal(ids[good[b:b + 60]], i) and torch.equal(dists[good[b:b + 60]], s)
    assert int(ids[list(special)].min()) >= -1 and int(ids.max()) < 909_300  # answers that mean nothing, in the index's range all the same
    ix.close()
