"""Searches at the sizes where the library's dispatch or its cut of the work changes, against the CPU oracle."""

import numpy as np
import pytest
import torch

from paper_2503_14649_b200 import synth
from tests.test_gpu_coarse_tc import _probe_parity
from tests.test_gpu_parity import _compare

pytestmark = pytest.mark.gpu


# Lists of tv vectors fill one tile of the scan.  nq, nprobe and k sit on both sides of the rules: a start of a query
# weighs on the shares or does not, at most 32 pairs or more, tables built with the selection or before it.
@pytest.mark.parametrize("M,tv,metric,nq,nprobe,k", [
    (16, 1024, "l2", 70, 10, 10), (32, 960, "l2", 16, 12, 20), (32, 960, "ip", 2, 16, 40), (48, 480, "l2", 90, 12, 100),
    (64, 960, "ip", 40, 12, 100), (64, 960, "l2", 3, 9, 33), (96, 384, "l2", 66, 12, 50), (128, 288, "ip", 20, 12, 64),
    (48, 480, "l2", 200, 1, 5)])
def test_scan_shares_and_tile_sizes(M, tv, metric, nq, nprobe, k):
    lengths = [0, 1, 31, tv - 1, tv, tv + 1, 2 * tv - 1, 2 * tv, 2 * tv + 1, 3 * tv + 33, 5 * tv + 1, 9 * tv, 0, tv // 2, 7, 4 * tv - 32]
    data = synth.make_ivfpq(sum(lengths), 2 * M if M < 128 else 128, len(lengths), M, nq, metric=metric, seed=M + nq)
    data.list_offsets = torch.tensor([0] + list(np.cumsum(lengths)), dtype=torch.int64)
    _compare(data, nprobe, k, max_probe_mismatch=1)


# Tensor-core coarse step: score matrix (nothing would be dropped), lists that overflow and are cut, and lists behind
# pilot thresholds with few and with many wanted entries.
@pytest.mark.parametrize("nlist,nq,nprobe,metric,bf16", [
    (255, 64, 32, "l2", False), (4097, 65, 32, "ip", True), (6000, 300, 100, "l2", False), (20_001, 1500, 20, "ip", True),
    (8192, 33, 24, "l2", True), (16_384, 70, 40, "ip", False), (32_768, 20, 300, "l2", True), (32_768, 17, 500, "ip", True)])
def test_coarse_candidates_by_list_count(nlist, nq, nprobe, metric, bf16):
    data = synth.make_ivfpq(2000, 64, nlist, 16, nq, metric=metric, seed=nlist + nq, coarse_bf16=bf16)
    _probe_parity(data, nprobe, 2)
