"""Queries with NaN, infinite or overflowing values: their own answers mean nothing, but every list and every id they get
belongs to the index, and the other queries of the batch are answered as if they were not there."""

import pytest
import torch

from paper_2503_14649_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _poison(q):
    """Rows 0 .. 4 of a batch: all NaN, one NaN, one +inf, one -inf, values whose products overflow."""
    p = q.clone()
    p[0] = float("nan")
    p[1, 7] = float("nan")
    p[2, 3] = float("inf")
    p[3, 5] = -float("inf")
    p[4] = 3.0e38
    return p


# fp32 scores; a score matrix of the tensor-core step; its candidate lists behind pilot thresholds and without; wide CTAs
# and narrow ones; the two-level quantiser
@pytest.mark.parametrize("nlist,nq,nprobe,metric,bf16,tree", [
    (300, 7, 12, "l2", False, 0), (300, 7, 300, "ip", True, 0), (255, 40, 32, "l2", True, 0), (8192, 40, 16, "l2", False, 0),
    (8192, 200, 40, "ip", True, 0), (20_001, 1500, 20, "l2", False, 0), (512, 6, 16, "l2", False, 32), (512, 6, 16, "ip", True, 32)])
def test_nonfinite_queries_leave_the_rest_of_the_batch_alone(nlist, nq, nprobe, metric, bf16, tree):
    data = synth.make_ivfpq(4000, 64, nlist, 16, nq, metric=metric, seed=nlist + nq, coarse_bf16=bf16)
    ix = binding.load_index_from(data, "cuda")
    if tree:
        level1 = data.centroids[:: nlist // tree].cuda().contiguous()
        offsets = torch.arange(0, nlist + 1, nlist // tree, dtype=torch.int32, device="cuda")
        ix.rago_index_set_coarse_tree(level1, offsets, 4)
    q = data.queries.cuda().contiguous()
    clean = ix.rago_search_probes(q, nprobe) + ix.rago_search(q, nprobe, 10)
    p = _poison(q)
    lists, coarse = ix.rago_search_probes(p, nprobe)
    ids, dists = ix.rago_search(p, nprobe, 10)
    torch.cuda.synchronize()
    ix.rago_check()
    for got, want in zip((lists, coarse, ids, dists), clean):
        assert torch.equal(got[5:], want[5:])
    assert bool((lists >= 0).all()) and bool((lists < nlist).all())
    assert all(len(set(row)) == nprobe for row in lists[:5].tolist())
    known = set(data.ids.tolist()) | {-1}
    assert set(ids[:5].flatten().tolist()) <= known
    ix.close()
