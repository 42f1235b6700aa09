"""Candidate buffers of the scan: groups of equal scores larger than a buffer, and values of k near its capacity."""

import pytest
import torch

from paper_2503_14649_b200 import binding

pytestmark = pytest.mark.gpu


def _scores(q, c, books, codes, metric):
    """Exact scores (smaller is better) of codes under one list with centroid c, in fp64."""
    M, _, dsub = books.shape
    out = torch.empty(q.shape[0], codes.shape[0], dtype=torch.float64, device=q.device)
    for i in range(q.shape[0]):
        r = (q[i] - c).double().view(M, 1, dsub)
        t = ((r - books.double()) ** 2).sum(2) if metric == "l2" else -(q[i].double().view(M, 1, dsub) * (books.double() + c.double().view(M, 1, dsub))).sum(2)
        out[i] = t[torch.arange(M, device=q.device)[None, :], codes.long()].sum(1)
    return out


# One list of mostly identical vectors, farther from the query than the few others among them: more equal scores than a buffer holds
# reach every CTA before the better ones do.  Sums of M fp32 terms: 1e-5 of the largest score covers their rounding.
@pytest.mark.parametrize("M,metric,nq,k", [(16, "l2", 1, 100), (32, "ip", 1, 33), (48, "l2", 1, 100), (64, "ip", 1, 100), (64, "l2", 1, 300), (80, "l2", 1, 40),
                                           (96, "l2", 1, 100), (96, "ip", 2, 500), (128, "ip", 1, 100), (64, "l2", 1, 10), (96, "l2", 70, 100)])
def test_better_vectors_behind_more_equal_ones_than_a_buffer_holds(M, metric, nq, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + k)
    N, d = 1_400_000, 4 * M
    c = torch.randn(1, d, generator=g, device="cuda")
    books = 0.3 * torch.randn(M, 256, 4, generator=g, device="cuda")
    q = (c + 0.3 * torch.randn(1, d, generator=g, device="cuda")).repeat(nq, 1).contiguous()
    every = torch.arange(256, device="cuda")[:, None].expand(256, M).to(torch.uint8)
    per_code = torch.stack([_scores(q[:1], c[0], books * (torch.arange(M, device="cuda") == m).view(M, 1, 1), every, metric)[0] for m in range(M)], 1)
    codes = per_code.argmax(0).to(torch.uint8).expand(N, M).contiguous()  # the worst code of every sub-space
    few = torch.randperm(N, generator=g, device="cuda")[:N // 1000]
    codes[few] = torch.randint(0, 256, (few.numel(), M), generator=g, device="cuda", dtype=torch.uint8)
    ix = binding.rago_index_load(c, books, codes, torch.tensor([0, N], device="cuda"), torch.arange(N, device="cuda"), metric)
    ids, dists = ix.rago_search(q, 1, k)
    torch.cuda.synchronize()
    ix.rago_check()
    exact = _scores(q[:1], c[0], books, codes[few], metric)[0]
    want, at = exact.sort()
    sign = 1.0 if metric == "l2" else -1.0
    for i in (0, nq - 1):
        assert torch.allclose(sign * dists[i].double(), want[:k], rtol=0, atol=1e-5 * float(want.abs().max()))
        assert set(ids[i].tolist()) <= set(few[at[:k + 5]].tolist())
    ix.close()


# Vectors from the farthest to the closest, over and over: nearly every one passes the threshold, the buffer is cut every few tiles, and what a
# cut keeps (up to k * 5 / 4 keys) has the tiles in flight pushed behind it.  Long enough that some cut meets the producer's look at the count.
@pytest.mark.parametrize("M,metric,k", [(16, "l2", 1024), (32, "ip", 1024), (48, "l2", 1000), (64, "ip", 1024), (80, "l2", 1024), (96, "l2", 1024),
                                        (96, "ip", 980), (96, "l2", 600), (128, "ip", 1024)])
def test_large_k_over_vectors_in_descending_order_of_score(M, metric, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + k)
    N, d, block = 2_000_000, 4 * M, 13_000
    c = torch.randn(1, d, generator=g, device="cuda")
    books = 0.3 * torch.randn(M, 256, 4, generator=g, device="cuda")
    q = (c + 0.3 * torch.randn(1, d, generator=g, device="cuda")).contiguous()
    codes = torch.randint(0, 256, (N, M), generator=g, device="cuda", dtype=torch.uint8)
    score = torch.cat([_scores(q, c[0], books, part, metric)[0] for part in codes.split(100_000)])
    order = torch.cat([b + score[b:b + block].argsort(descending=True) for b in range(0, N, block)])
    codes, score = codes[order].contiguous(), score[order]
    ix = binding.rago_index_load(c, books, codes, torch.tensor([0, N], device="cuda"), torch.arange(N, device="cuda"), metric)
    want, at = score.sort()
    allowed = set(at[:k + 8].tolist())
    sign = 1.0 if metric == "l2" else -1.0
    for _ in range(10):
        ids, dists = ix.rago_search(q, 1, k)
        torch.cuda.synchronize()
        ix.rago_check()
        assert torch.allclose(sign * dists[0].double(), want[:k], rtol=0, atol=1e-5 * float(want.abs().max()))
        assert set(ids[0].tolist()) <= allowed
    ix.close()


# Row groups of 48-byte tiles are dealt over the warps: lists that end on, before and behind a group, a round of 15 groups and a tile of 960.
@pytest.mark.parametrize("metric,k", [("l2", 100), ("ip", 10), ("l2", 1)])
def test_lists_around_the_row_groups_of_a_48_byte_tile(metric, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(48 + k)
    sizes = [1, 31, 32, 33, 64, 65, 479, 480, 481, 511, 513, 928, 959, 960, 961, 1439, 1440, 1441, 1920, 1953]
    nlist, N, M = len(sizes), sum(sizes), 48
    c = torch.randn(nlist, 4 * M, generator=g, device="cuda")
    books = 0.3 * torch.randn(M, 256, 4, generator=g, device="cuda")
    codes = torch.randint(0, 256, (N, M), generator=g, device="cuda", dtype=torch.uint8)
    offsets = torch.tensor([0] + sizes, device="cuda").cumsum(0)
    ix = binding.rago_index_load(c, books, codes, offsets, torch.arange(N, device="cuda"), metric)
    q = torch.randn(20, 4 * M, generator=g, device="cuda")
    sign = 1.0 if metric == "l2" else -1.0
    for nprobe in (1, nlist):  # a query's own list alone (its last vectors among the results), and all of them
        near = (c + 0.1 * q).contiguous()
        ids, dists = ix.rago_search(near, nprobe, k)
        torch.cuda.synchronize()
        ix.rago_check()
        lists, _ = ix.rago_search_probes(near, nprobe)
        for i in range(nlist):
            score = torch.full((N,), float("inf"), dtype=torch.float64, device="cuda")
            for l in lists[i].tolist():
                a, b = int(offsets[l]), int(offsets[l + 1])
                score[a:b] = _scores(near[i:i + 1], c[l], books, codes[a:b], metric)[0]
            want, at = score.sort()
            n = min(k, int(torch.isfinite(score).sum()))
            assert torch.allclose(sign * dists[i, :n].double(), want[:n], rtol=0, atol=1e-5 * float(want[:n].abs().max()))
            assert set(ids[i, :n].tolist()) <= set(at[:n + 5].tolist())
    ix.close()


# Few 46 KB tiles are cut into tiles of 256 vectors: lists around that size, and as many probes as leave whole tiles (of 74 CTAs' worth) on either side.
@pytest.mark.parametrize("M,nq,nprobe,k", [(96, 1, 20, 100), (48, 1, 20, 100), (96, 3, 20, 10), (48, 2, 11, 300), (96, 3, 5, 1), (48, 4, 20, 7), (96, 10, 10, 50)])
def test_few_tiles_are_smaller(M, nq, nprobe, k):
    g = torch.Generator(device="cuda")
    g.manual_seed(M + nq)
    sizes = [1, 31, 255, 256, 257, 479, 480, 481, 511, 512, 513, 767, 768, 769, 959, 960, 961, 1023, 1024, 1025]
    N, nlist = sum(sizes), len(sizes)
    c = torch.randn(nlist, 4 * M, generator=g, device="cuda")
    books = 0.3 * torch.randn(M, 256, 4, generator=g, device="cuda")
    codes = torch.randint(0, 256, (N, M), generator=g, device="cuda", dtype=torch.uint8)
    offsets = torch.tensor([0] + sizes, device="cuda").cumsum(0)
    ix = binding.rago_index_load(c, books, codes, offsets, torch.arange(N, device="cuda"), "l2")
    q = torch.randn(nq, 4 * M, generator=g, device="cuda")
    ids, dists = ix.rago_search(q, nprobe, k)
    torch.cuda.synchronize()
    ix.rago_check()
    lists, _ = ix.rago_search_probes(q, nprobe)
    for i in range(nq):
        score = torch.full((N,), float("inf"), dtype=torch.float64, device="cuda")
        for l in lists[i].tolist():
            a, b = int(offsets[l]), int(offsets[l + 1])
            score[a:b] = _scores(q[i:i + 1], c[l], books, codes[a:b], "l2")[0]
        want, at = score.sort()
        n = min(k, int(torch.isfinite(score).sum()))
        assert torch.allclose(dists[i, :n].double(), want[:n], rtol=0, atol=1e-5 * float(want[:n].abs().max()))
        assert set(ids[i, :n].tolist()) <= set(at[:n + 5].tolist())
    ix.close()
