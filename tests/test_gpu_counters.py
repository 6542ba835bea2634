"""Work counters beyond 32 bits: one tile whose warp takes more than 2^32
distances."""
import numpy as np
import pytest
import torch

from paper_2112_10408_gb300 import tnn

pytestmark = pytest.mark.gpu


def test_pairs_of_one_warp_pass_32_bits():
    # Segments of 64 points that jump between x = -100 and 100: every axis
    # passes by the queries, so every segment's bound is zero and all of its
    # points, far away, are scanned.  32 queries, one tile, one warp; their
    # neighbours are the last segment's.
    S, k = (1 << 21) + 4, 4
    n = 64 * S
    x = torch.zeros((n, 4), device="cuda")
    x[0::2, 0], x[1::2, 0] = 100.0, -100.0
    x[:, 3] = torch.arange(n, device="cuda") >> 6
    x[-64:, 0] = torch.arange(64, device="cuda") / 64.0
    q = torch.zeros((32, 4), device="cuda")
    q[:, 3] = 2.0 * S
    ix = tnn.tnn_build_segments(x, np.array([0, n], np.int64), (1.0, 1.0, 1.0, 0.0), 64)
    idx, _, st = tnn.tnn_knn(ix, k, 0.0, q=q, stats=True, defer_cells=-1.0)
    assert idx.cpu().tolist() == [[n - 64, n - 63, n - 62, n - 61]] * 32
    assert st["pairs"] == 32 * n and n * 32 > 1 << 32
    assert st["segs_scanned"] == 32 * S
    ix.destroy()
    tnn.tnn_memory_trim()
