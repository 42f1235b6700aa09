"""Searches at the sizes where the library's dispatch or its cut of the work changes, against the CPU oracle."""

import numpy as np
import pytest
import torch

from paper_2503_14649_b200 import binding, synth
from tests.test_gpu_coarse_tc import _probe_parity
from tests.test_gpu_parity import _compare

pytestmark = pytest.mark.gpu


# Lists of tv vectors fill one tile of the scan.  nq, nprobe and k sit on both sides of the rules: at most 32 pairs or
# more, tables built with the selection or before it; the start of a query weighs on the shares with 16 bytes, 70 queries and
# with 64 bytes, 40 queries only (test_scan_shares_with_weighted_query_starts has the other sizes).
@pytest.mark.parametrize("M,tv,metric,nq,nprobe,k", [
    (16, 1024, "l2", 70, 10, 10), (32, 960, "l2", 16, 12, 20), (32, 960, "ip", 2, 16, 40), (48, 480, "l2", 90, 12, 100),
    (64, 960, "ip", 40, 12, 100), (64, 960, "l2", 3, 9, 33), (96, 384, "l2", 66, 12, 50), (128, 288, "ip", 20, 12, 64),
    (48, 480, "l2", 200, 1, 5)])
def test_scan_shares_and_tile_sizes(M, tv, metric, nq, nprobe, k):
    lengths = [0, 1, 31, tv - 1, tv, tv + 1, 2 * tv - 1, 2 * tv, 2 * tv + 1, 3 * tv + 33, 5 * tv + 1, 9 * tv, 0, tv // 2, 7, 4 * tv - 32]
    data = synth.make_ivfpq(sum(lengths), 2 * M if M < 128 else 128, len(lengths), M, nq, metric=metric, seed=M + nq)
    data.list_offsets = torch.tensor([0] + list(np.cumsum(lengths)), dtype=torch.int64)
    _compare(data, nprobe, k, max_probe_mismatch=1)


def _with_lengths(lengths, M, nq, metric, seed):
    data = synth.make_ivfpq(sum(lengths), 2 * M if M < 128 else 128, len(lengths), M, nq, metric=metric, seed=seed)
    data.list_offsets = torch.tensor([0] + list(np.cumsum(lengths)), dtype=torch.int64)
    return data


def _lead(data, nq, nprobe, k):
    ix = binding.load_index_from(data, "cuda")
    lead = ix.rago_debug_search_plan(nq, nprobe, k)["lead"]
    ix.close()
    return lead


# Every code size where the start of a query weighs on the shares: up to 32 pairs (a few long lists) and more, the weight of
# small k, of a 64 KB table and of a 128 KB one.
@pytest.mark.parametrize("M,tv,nlist,tiles,metric,nq,nprobe,k", [
    (16, 1024, 8, 34, "l2", 4, 8, 10), (64, 960, 8, 17, "ip", 4, 8, 20), (32, 960, 16, 6, "l2", 16, 12, 20),
    (48, 480, 16, 3, "l2", 90, 12, 100), (64, 960, 16, 4, "ip", 70, 12, 100), (80, 256, 16, 5, "l2", 60, 12, 100),
    (96, 384, 16, 4, "ip", 66, 12, 50), (96, 384, 8, 25, "l2", 4, 8, 10), (128, 288, 16, 4, "l2", 66, 12, 64)])
def test_scan_shares_with_weighted_query_starts(M, tv, nlist, tiles, metric, nq, nprobe, k):
    ragged = [(-1) ** l * ((37 * l) % tv) for l in range(nlist)]  # longer and shorter than the average in turn
    lengths = [tiles * tv + r for r in ragged]
    data = _with_lengths(lengths, M, nq, metric, seed=M + nq)
    assert _lead(data, nq, nprobe, k) > 0
    _compare(data, nprobe, k, max_probe_mismatch=1)


# All vectors in one list, so that most probed lists are empty although the average is long: shares that lie in the starts of
# queries have no tile, and some queries have no candidate at all.
@pytest.mark.parametrize("M,tv,nlist,total,nq,nprobe,k", [
    (16, 1024, 16, 34, 8, 4, 10), (16, 1024, 64, 4, 100, 4, 10), (64, 960, 64, 4, 100, 4, 100), (96, 384, 64, 8, 100, 4, 10),
    (16, 1024, 64, 4, 100, 1, 10)])
@pytest.mark.parametrize("full", [0, -1])
def test_scan_shares_without_a_tile(M, tv, nlist, total, nq, nprobe, k, full):
    lengths = [0] * nlist
    lengths[full] = nlist * total * tv
    data = _with_lengths(lengths, M, nq, "ip", seed=M + nlist)
    if nprobe > 1:
        assert _lead(data, nq, nprobe, k) > 0
    _compare(data, nprobe, k, max_probe_mismatch=1)


# Tensor-core coarse step: score matrix (nothing would be dropped; 4097, 6000 lists), lists that overflow and are cut (20 001), and
# lists behind pilot thresholds with few and with many wanted entries.
@pytest.mark.parametrize("nlist,nq,nprobe,metric,bf16", [
    (255, 64, 32, "l2", False), (4097, 65, 32, "ip", True), (6000, 300, 100, "l2", False), (20_001, 1500, 20, "ip", True),
    (8192, 33, 24, "l2", True), (16_384, 70, 40, "ip", False), (32_768, 20, 300, "l2", True), (32_768, 17, 500, "ip", True)])
def test_coarse_candidates_by_list_count(nlist, nq, nprobe, metric, bf16):
    data = synth.make_ivfpq(2000, 64, nlist, 16, nq, metric=metric, seed=nlist + nq, coarse_bf16=bf16)
    _probe_parity(data, nprobe, 2)
