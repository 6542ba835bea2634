"""The warp-per-query kernel where it can go wrong: list registers around
their limits, long chains of equal distances, more candidates than slots, and
queries whose neighbours lie in other cells than their own.  Every query is
handed over (a deferral radius of nearly zero); indices are bit-exact against
the FP64 oracle, distances within 1e-5 relative."""
import numpy as np
import pytest
import torch

import oracle
from paper_2112_10408_gb300 import synth
from paper_2112_10408_gb300 import tnn
from tests._helpers import assert_knn_equal

pytestmark = pytest.mark.gpu
SIG = synth.SIGMA_DEFAULT


def _check(wl, K, k, lag=0.0, q=None, sigma=SIG, what="", defer=1e-6):
    ix = tnn.tnn_build_segments(torch.from_numpy(wl.xyzt).cuda(), wl.traj_off, sigma, K)
    qd = None if q is None else torch.from_numpy(q).cuda()
    gi, gd, st = tnn.tnn_knn(ix, k, lag, q=qd, defer_cells=defer, stats=True)
    oi, od = oracle.knn(wl.xyzt, k, sigma, lag=lag, queries=q)
    assert_knn_equal(gi.cpu().numpy(), gd.cpu().numpy(), oi, od, what=what)
    return st


@pytest.mark.parametrize("k", [1, 4, 15, 16, 17, 31, 32, 33, 63, 64])
def test_list_registers_around_their_limits(k):
    wl = synth.flights(31, 47, seed=400 + k, n_routes=4)
    st = _check(wl, 9, k, what=f"k={k}")
    assert st["warp_queries"] > 0.9 * wl.n
    _check(wl, 9, k, lag=200.0, what=f"k={k} lag")


@pytest.mark.parametrize("copies", [3, 11, 30])
def test_chains_of_equal_distances(copies):
    # every sample `copies` times at the same place and time: chains as long
    # as that, settled by index
    rng = np.random.default_rng(copies)
    base = np.sort(rng.uniform(0.0, 40.0, (60, 4)), axis=0)
    xyzt = np.repeat(base, copies, axis=0).astype(np.float32)
    n = xyzt.shape[0]
    off = np.array([0, n // 3, n], np.int64)
    wl = synth.Workload(xyzt, np.zeros((n, 2), np.float32), off, np.zeros(n, np.int32), "copies")
    for k in (5, 16, 32, 64):
        _check(wl, 10, k, what=f"{copies} copies k={k}")
        _check(wl, 10, k, what=f"{copies} copies k={k} tiles", defer=-1.0)


def test_more_candidates_than_slots():
    # points ordered so that later ones are nearer to the queries: nearly
    # every one passes and the slots are renumbered
    rng = np.random.default_rng(3)
    n = 6000
    xyzt = rng.uniform(0.0, 2.0, (n, 4)).astype(np.float32)
    xyzt[:, 0] = np.linspace(0.0, 50.0, n)
    xyzt[:, 3] = np.arange(n) * 0.01
    wl = synth.Workload(xyzt, np.zeros((n, 2), np.float32), np.array([0, n], np.int64), np.zeros(n, np.int32),
                        "approach")
    q = rng.uniform(0.0, 2.0, (40, 4)).astype(np.float32)
    q[:, 0] = rng.uniform(0.0, 52.0, 40)
    q[:, 3] = 1e4
    for k in (16, 64):
        _check(wl, 64, k, q=q, sigma=(1.0, 1.0, 1.0, 1e-12), what=f"approach k={k}")


def test_neighbours_in_far_cells():
    # two groups far apart in space and time: queries of the second find too
    # few points near them and must reach across many cells and buckets
    a = synth.flights(30, 60, seed=71, n_routes=3)
    b = synth.flights(2, 40, seed=72, n_routes=1)
    x2 = b.xyzt.copy()
    x2[:, 0] += 9000.0
    x2[:, 3] += 4000.0
    xyzt = np.concatenate([a.xyzt, x2]).astype(np.float32)
    off = np.concatenate([a.traj_off, a.n + b.traj_off[1:]])
    n = xyzt.shape[0]
    wl = synth.Workload(xyzt, np.zeros((n, 2), np.float32), off, np.zeros(n, np.int32), "far")
    for k, defer in ((32, 0.0), (64, 1e-6)):
        _check(wl, 12, k, what=f"far k={k}", defer=defer)
