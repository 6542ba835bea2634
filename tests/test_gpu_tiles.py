"""The grid tile kernel where it can go wrong: list lengths around its classes
(8, 16, 32, 64) and rows that are or are not whole 16-byte words, tiles whose
queries lie apart, tiles that see more candidates than they have slots for,
and windows of every class in one batch.  Neighbour indices are bit-exact
against the FP64 oracle, distances within 1e-5 relative."""
import numpy as np
import pytest
import torch

import oracle
from paper_2112_10408_gb300 import synth
from paper_2112_10408_gb300 import tnn
from tests._helpers import assert_knn_equal

pytestmark = pytest.mark.gpu
SIG = synth.SIGMA_DEFAULT


def _index(wl, K, sigma=SIG):
    return tnn.tnn_build_segments(torch.from_numpy(wl.xyzt).cuda(), wl.traj_off, sigma, K)


def _check(ix, wl, k, lag=0.0, q=None, sigma=SIG, what="", **kw):
    qd = None if q is None else torch.from_numpy(q).cuda()
    gi, gd = tnn.tnn_knn(ix, k, lag, q=qd, **kw)
    torch.cuda.synchronize()
    oi, od = oracle.knn(wl.xyzt, k, sigma, lag=lag, queries=q)
    assert_knn_equal(gi.cpu().numpy(), gd.cpu().numpy(), oi, od, what=what)


def _dense(n, seed, side=3.0):
    """Points uniform in a small box and in time, in sets of 40."""
    rng = np.random.default_rng(seed)
    xyzt = rng.uniform(0.0, side, (n, 4)).astype(np.float32)
    xyzt[:, 3] = np.sort(rng.uniform(0.0, 600.0, n).astype(np.float32))
    off = np.append(np.arange(0, n, 40), n).astype(np.int64)
    return synth.Workload(xyzt, np.zeros((n, 2), np.float32), off, np.zeros(n, np.int32), "dense")


@pytest.mark.parametrize("k", [1, 2, 7, 8, 9, 12, 15, 16, 17, 31, 32, 33, 63, 64])
def test_list_lengths_around_the_classes(k):
    wl = synth.flights(37, 61, seed=300 + k, n_routes=4)
    ix = _index(wl, 11)
    _check(ix, wl, k, what=f"k={k}")
    _check(ix, wl, k, lag=90.0, what=f"k={k} never deferred", defer_cells=-1.0)


@pytest.mark.parametrize("k", [8, 32])
def test_rows_that_are_not_16_byte_aligned(k):
    wl = synth.flights(20, 45, seed=7, n_routes=3)
    ix = _index(wl, 9)
    bi = torch.full((wl.n * k + 1,), -7, dtype=torch.int32, device="cuda")
    bd = torch.full((wl.n * k + 1,), -7.0, dtype=torch.float32, device="cuda")
    out = bi[1:].view(wl.n, k), bd[1:].view(wl.n, k)
    tnn.tnn_knn(ix, k, 0.0, out=out)
    torch.cuda.synchronize()
    oi, od = oracle.knn(wl.xyzt, k, SIG)
    assert_knn_equal(out[0].cpu().numpy(), out[1].cpu().numpy(), oi, od, what="unaligned rows")
    assert bi[0].item() == -7 and bd[0].item() == -7.0


@pytest.mark.parametrize("k", [5, 64])
@pytest.mark.parametrize("defer", [0.0, 0.4, -1.0])
def test_tiles_with_more_candidates_than_slots(k, defer):
    # Queries in no order over dense points, late enough that thousands of
    # points pass while the lists converge; at k = 64 the 32 lists of a tile
    # hold more distinct points than the slot table.
    wl = _dense(12000, 5)
    rng = np.random.default_rng(6)
    q = rng.uniform(0.0, 3.0, (509, 4)).astype(np.float32)
    q[:, 3] = rng.uniform(550.0, 700.0, 509)
    sigma = (1.0, 1.0, 1.0, 1e-9)
    _check(_index(wl, 40, sigma), wl, k, q=q, sigma=sigma, what=f"dense k={k}", defer_cells=defer)


@pytest.mark.parametrize("defer", [0.0, -1.0])
def test_tiles_whose_queries_lie_apart(defer):
    # runs of 1 to 9 neighbouring queries, far from one another, in one array;
    # some before every point, one so far away that its FP32 distances overflow
    wl = synth.flights(120, 90, seed=31, n_routes=9)
    rng = np.random.default_rng(8)
    rows = np.concatenate([np.arange(r, r + n) for r, n in zip(rng.integers(0, wl.n - 9, 60),
                                                               rng.integers(1, 10, 60))])
    q = wl.xyzt[rows].copy()
    q[::13, 3] = -5.0
    q[20, 0] = 1e25
    _check(_index(wl, 15), wl, 20, lag=30.0, q=q, what="runs of queries", defer_cells=defer)


def test_duplicates_and_ties_in_every_class():
    wl = synth.lattice(24, 40, seed=9, side=4)
    ix = _index(wl, 8)
    for k in (3, 8, 16, 32, 64):
        _check(ix, wl, k, what=f"lattice k={k}")


def test_batch_of_every_class():
    wls = [synth.flights(12 + 5 * i, 41 + i, seed=50 + i, n_routes=3) for i in range(7)]
    ks = [64, 3, 32, 16, 9, 33, 8]
    ixs = [_index(wl, 10) for wl in wls]
    b = tnn.Batch(ixs, ks)
    for _ in range(2):
        b.run()
    st = b.stats()
    assert st["queries"] == sum(wl.n for wl in wls)
    for wl, k, gi, gd in zip(wls, ks, b.idx, b.d2):
        oi, od = oracle.knn(wl.xyzt, k, SIG)
        assert_knn_equal(gi.cpu().numpy(), gd.cpu().numpy(), oi, od, what=f"window k={k}")
