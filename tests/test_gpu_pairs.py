"""Queries that share long lists are scanned two at a time (pair.cuh).  The answers have to be those of the scan of one query, bit
for bit: the same queries are searched in batches of 64, which are too small for pairs."""

from types import SimpleNamespace

import numpy as np
import pytest
import torch

import oracle
from paper_2503_14649_b200 import binding
from tests.helpers import IvfPqRescorer, host_index, match_results

pytestmark = pytest.mark.gpu


def _index(M, dsub, sizes, metric="l2", bf16=False, seed=0, same_codes=False):
    """Lists of the given sizes around random centroids; random codes (or one code throughout)."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    nlist, N, d = len(sizes), sum(sizes), M * dsub
    c = torch.randn(nlist, d, generator=g, device="cuda")
    books = 0.3 * torch.randn(M, 256, dsub, generator=g, device="cuda")
    codes = torch.randint(0, 256, (N, M), generator=g, device="cuda", dtype=torch.uint8)
    if same_codes:
        codes[:] = codes[:1]
    offsets = torch.tensor([0] + list(np.cumsum(sizes)), device="cuda", dtype=torch.int64)
    ids = torch.randperm(N, generator=g, device="cuda")
    ix = binding.rago_index_load(c.bfloat16() if bf16 else c, books, codes, offsets, ids, metric)
    return ix, c, (c.bfloat16() if bf16 else c, books, codes, offsets, ids)


def _queries(c, owners, seed=1):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return (c[torch.tensor(owners, device="cuda")] + 0.3 * torch.randn(len(owners), c.shape[1], generator=g, device="cuda")).contiguous()


def _launches(ix, q, nprobe, k):
    n = binding.rago_kernel_launches()
    ids, dists = ix.rago_search(q, nprobe, k)
    torch.cuda.synchronize()
    ix.rago_check()
    return binding.rago_kernel_launches() - n, ids, dists


def _check(ix, q, nprobe, k, ids_too=True):
    launches, ids, dists = _launches(ix, q, nprobe, k)
    # the same call without pairs (k above their limit): the same launches but five
    assert launches == _launches(ix, q, nprobe, 1024)[0] + 5
    for b in range(0, q.shape[0], 64):
        part = q[b:b + 64].contiguous()
        i, s = ix.rago_search(part, nprobe, k)
        assert torch.equal(dists[b:b + 64].view(torch.int32), s.view(torch.int32)), b
        if ids_too:
            assert torch.equal(ids[b:b + 64], i), b
    return ids, dists


# Long lists around the tiles' sizes (480 and 960 vectors), small and empty ones beside them; an odd number of queries on the longest list
# leaves one single; 40 probes make more than 64 entries a pair.
@pytest.mark.parametrize("M,dsub,metric,bf16,nq,nprobe,k", [
    (96, 4, "l2", False, 101, 8, 100), (96, 8, "ip", True, 130, 40, 10), (64, 4, "l2", True, 160, 12, 100), (64, 8, "ip", False, 129, 40, 512),
    (48, 4, "l2", False, 200, 9, 1), (48, 16, "ip", False, 131, 33, 300), (32, 4, "l2", False, 250, 12, 20), (32, 8, "ip", True, 300, 5, 64),
    (16, 8, "l2", False, 333, 12, 33), (16, 4, "ip", False, 301, 1, 100), (96, 4, "l2", False, 70, 1, 512)])
def test_pairs_answer_as_single_queries_do(M, dsub, metric, bf16, nq, nprobe, k):
    big = 300_000_000 // (M * nq)  # enough work that the host looks for pairs
    sizes = [7 * big + 1, 4 * big, 960, 961, 959, 480, 481, 479, 1, 0, 31, 33] + [big // 64 + i for i in range(40)]
    ix, c, arrays = _index(M, dsub, sizes, metric, bf16, seed=M + nq)
    owners = [0] * (nq // 2 | 1) + [1] * (nq // 4) + [(3 * i) % len(sizes) for i in range(nq)]
    q = _queries(c, owners[:nq])
    ids, dists = _check(ix, q, nprobe, k)
    # and a few of them as the oracle does
    host = host_index(oracle, SimpleNamespace(metric=metric, **dict(zip(("centroids", "codebooks", "codes", "list_offsets", "ids"), arrays))))
    some, sign = [0, 1, nq // 2, nq - 1], 1.0 if metric == "l2" else -1.0
    oi, od = oracle.ivfpq_search(host, q[some].cpu().numpy(), nprobe, k)
    rescore = IvfPqRescorer(oracle, host)
    for n, s in enumerate(some):
        assert not match_results(ids[s].cpu().numpy(), sign * dists[s].cpu().numpy(), oi[n], sign * od[n], rel=1e-4,
                                 rescore=rescore.for_query(q[s].cpu().numpy(), sign)), s
    ix.close()


# Every vector of a list has the same code: all bounds of a tile are equal and pass together, so the buffers are made exact on the way
# (which of the equal vectors are returned is open).  With one far code beside them the 16-bit halves are as coarse as they get.
@pytest.mark.parametrize("M,k", [(96, 100), (48, 10), (64, 512), (32, 1), (16, 40)])
def test_pairs_with_more_equal_scores_than_a_buffer_holds(M, k):
    sizes = [16_000_000 // M, 3000, 2000, 500]
    ix, c, _ = _index(M, 4, sizes, seed=M, same_codes=True)
    _check(ix, _queries(c, [0] * 60 + [1, 2, 3] * 3 + [0] * 31), 3, k, ids_too=False)
    ix.close()


# A workspace sized for a larger k, more probes or more queries than pairs go with serves fewer of them, with pairs.
@pytest.mark.parametrize("nq,nprobe,k", [(128, 3, 1024), (128, 4, 100), (300, 3, 100), (5000, 4, 1024)])
def test_a_larger_workspace_serves_a_call_with_pairs(nq, nprobe, k):
    ix, c, _ = _index(64, 4, [900_000, 5000, 4000, 300], seed=6)
    q = _queries(c, [0] * 90 + [1] * 38)
    ws = torch.empty(ix.search_workspace_bytes(nq, nprobe, k), dtype=torch.uint8, device="cuda")
    n = binding.rago_kernel_launches()
    ids, dists = ix.rago_search(q, 3, 100, workspace=ws)
    n = binding.rago_kernel_launches() - n
    torch.cuda.synchronize()
    assert n == _launches(ix, q, 3, 1024)[0] + 5
    i, s = ix.rago_search(q[:64].contiguous(), 3, 100)
    assert torch.equal(ids[:64], i) and torch.equal(dists[:64], s)
    ix.close()


# Queries whose tables are not bounded have no partner; the others' answers do not change.
def test_queries_with_infinite_and_huge_values_have_no_partner():
    ix, c, _ = _index(64, 4, [900_000, 5000, 4000, 300], seed=5)
    q = _queries(c, [0] * 80 + [1] * 17)
    q[3, 5] = float("inf")
    q[10] = float("nan")
    q[11, 0] = 3e38
    q[40] *= 1e30
    _, ids, dists = _launches(ix, q, 3, 50)
    good = [i for i in range(97) if i not in (3, 10, 11, 40)]
    i, s = ix.rago_search(q[good][:64].contiguous(), 3, 50)
    assert torch.equal(ids[good][:64], i) and torch.equal(dists[good][:64], s)
    ix.close()
