"""Flat search's final selection alone, over lists that a search does not leave in a test."""

import pytest
import torch

from paper_2503_14649_b200 import binding, synth

pytestmark = pytest.mark.gpu


def _lists(scores):
    """Raw entries [nq, nlists, stride] over scores of that shape; row numbers follow the storage order."""
    nq, nlists, stride = scores.shape
    rows = torch.arange(nlists * stride, dtype=torch.int64, device=scores.device).view(1, nlists, stride).expand(nq, -1, -1)
    return (scores.contiguous().view(torch.int32).long() << 32) | rows


def _check(scores, counts, k):
    """The k best of the entries below each list's count, equal scores by row number."""
    nq, nlists, stride = scores.shape
    ids, got = binding.rago_selftest_final_selection(counts, _lists(scores).contiguous(), k)
    torch.cuda.synchronize()
    taken = torch.arange(stride, device=scores.device).view(1, 1, -1) < counts.clamp(0, stride).unsqueeze(2)
    flat = torch.where(taken, scores, torch.full_like(scores, -float("inf"))).view(nq, -1)
    want, rows = flat.sort(dim=1, descending=True, stable=True)
    m = min(k, flat.shape[1])
    valid = torch.arange(m, device=scores.device).view(1, -1) < taken.view(nq, -1).sum(1, keepdim=True)
    assert torch.equal(got[:, :m], want[:, :m])
    assert torch.equal(ids[:, :m], torch.where(valid, rows[:, :m], torch.full_like(rows[:, :m], -1)))
    assert bool((ids[:, m:] == -1).all()) and bool(torch.isneginf(got[:, m:]).all())


def _normal(*shape, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda")


# An expired wait ends a search with an error word, and the readers of its lists must stay inside them whatever the
# count words hold (a search that reads past its lists would take the GPU's context down instead).
@pytest.mark.parametrize("nlists,stride,k", [(1, 512, 10), (296, 512, 100), (600, 40, 300), (3, 1024, 1024)])
def test_count_words_that_no_kernel_wrote_stay_inside_the_lists(nlists, stride, k):
    scores = _normal(4, nlists, stride, seed=nlists)
    counts = torch.randint(0, stride + 1, (4, nlists), dtype=torch.int32, device="cuda")
    for i, v in enumerate((-1, -(2 ** 31), 2 ** 31 - 1, stride + 1, 0x7F7F7F7F, 0)):
        counts.view(-1)[i::7] = v
    counts[3] = -5
    _check(scores, counts, k)


# A list's entries ascend, descend or stand in any order, so that what the first entries say about the rest holds or does
# not: the rest is streamed past their bound, streamed in vain, or taken in rounds; a last group of lists may be empty.
@pytest.mark.parametrize("nlists,stride,k", [(296, 512, 1), (296, 512, 10), (296, 896, 400), (100, 1024, 960), (40, 256, 300), (520, 64, 100)])
@pytest.mark.parametrize("order", ["random", "ascending", "descending", "equal"])
def test_final_selection_over_many_entries_in_any_order(nlists, stride, k, order):
    scores = _normal(3, nlists, stride, seed=k)
    if order in ("ascending", "descending"):
        scores = scores.view(3, -1).sort(dim=1, descending=order == "descending")[0].view(3, nlists, stride)
    elif order == "equal":
        scores = (scores * 2).round()  # a few values, thousands of rows each
    counts = torch.full((3, nlists), stride, dtype=torch.int32, device="cuda")
    counts[1, ::3] = 0
    counts[2, 512:] = 0
    _check(scores.contiguous(), counts, k)


# k beyond the fused selection: panels on the fp32 pipes, one chunk of rows (its keys are the answer) or two; k above N.
@pytest.mark.parametrize("N,k", [(900, 1024), (1, 961), (3000, 1000), (65_536, 1024), (65_537, 961)])
def test_flat_search_beyond_the_fused_selection(N, k):
    db, q = synth.make_flat(N, 64, 20, seed=N, device="cuda")
    ids, scores = binding.rago_flat_search(db, q, k)
    exact = q.double() @ db.double().T
    m = min(k, N)
    want, _ = exact.topk(m, 1)
    assert torch.allclose(scores[:, :m].double(), want, rtol=0, atol=64 * 2.0 ** -24)  # 64 products of unit-norm rows in fp32
    assert torch.allclose(exact.gather(1, ids[:, :m]), want, rtol=0, atol=64 * 2.0 ** -24)
    assert all(len(set(row)) == m for row in ids[:, :m].tolist())
    assert bool((ids[:, m:] == -1).all()) and bool(torch.isneginf(scores[:, m:]).all())
