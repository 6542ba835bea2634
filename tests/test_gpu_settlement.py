"""Settlement of the grid tile kernel's lists where the truncated keys order
candidates otherwise than their distances: neighbours are those of the FP64
oracle, bit for bit."""
import numpy as np
import pytest
import torch

import oracle
from paper_2112_10408_gb300 import synth
from paper_2112_10408_gb300 import tnn
from tests._helpers import assert_knn_equal

pytestmark = pytest.mark.gpu
SIG = (1.0, 1.0, 10.0, 0.01)


def _run(xyzt, off, q, k, sigma, K=20, what="", **kw):
    ix = tnn.tnn_build_segments(torch.from_numpy(xyzt).cuda(), off, sigma, K)
    gi, gd, st = tnn.tnn_knn(ix, k, 0.0, q=torch.from_numpy(q).cuda(), stats=True, **kw)
    oi, od = oracle.knn(xyzt, k, sigma, queries=q)
    assert_knn_equal(gi.cpu().numpy(), gd.cpu().numpy(), oi, od, what=what)
    return st


@pytest.mark.parametrize("defer", [0.0, -1.0])
def test_last_listed_row_is_not_the_farthest_of_the_first_k(defer):
    # rank 8 is point 0; its FP32 distance is a few units above the start of
    # the bucket after that of point 1, and point 6 lies beside it
    rows = """-0x1.7789dep+2 0x1.dec9cep-1 0x1.404b9p+3 0x1.ef279cp+9
        0x1.ab38f6p+1 0x1.fbb4f6p+2 0x1.453abcp+3 0x1.efae6cp+9
        -0x1.8c044ap+2 -0x1.b19dfap+0 0x1.453ffp+3 0x1.f00988p+9
        -0x1.de57bap+0 -0x1.2e643ep+3 0x1.42158ep+3 0x1.f03ce4p+9
        0x1.c2adfep+2 -0x1.454e06p+3 0x1.4180bp+3 0x1.f06db2p+9
        0x1.94d246p+3 -0x1.4a3d56p+1 0x1.413c2p+3 0x1.f0a31ap+9
        -0x1.50314ap+2 0x1.54986ap+1 0x1.42c9c4p+3 0x1.f13306p+9
        0x1.982accp+2 -0x1.3e6cf6p+0 0x1.404b1ap+3 0x1.f20da4p+9
        0x1.4e60dcp+2 0x1.d02f78p+0 0x1.40d1dep+3 0x1.f24acp+9
        0x1.3c383p+0 0x1.3d5d6p+1 0x1.4185p+3 0x1.f2907ap+9
        -0x1.b7fa66p+0 -0x1.0a9d5p+0 0x1.423848p+3 0x1.f2d692p+9
        -0x1.2aecdep-2 -0x1.6abc86p+2 0x1.424c2ep+3 0x1.f3174p+9
        0x1.54b316p+2 -0x1.c274ap+2 0x1.40f1ep+3 0x1.f3513ap+9"""
    xyzt = np.array([[float.fromhex(v) for v in r.split()] for r in rows.splitlines()], np.float32)
    q = np.tile(np.array([[3.25, -1.5, 10.0, 1000.0]], np.float32), (3, 1))
    _run(xyzt, np.array([0, 13], np.int64), q, 8, SIG, what="13 points", defer_cells=defer)


def _clusters(k, n, seed):
    """n groups of points around three copies of a query each, 1,000 s apart:
    k - 2 near ones, two in one bucket of the truncated keys (one at its top,
    one near its bottom), eight in the next (one at its start), in any order."""
    rng = np.random.default_rng(seed)
    slots = 1024 if k > 32 else 512
    pts, off, qs = [], [0], []
    for i in range(n):
        base = np.float32(rng.uniform(70.0, 120.0))
        edge = (int(base.view(np.int32)) // slots + 1) * slots
        ulp = float(np.spacing(base))
        edge = float(np.int32(edge).view(np.float32))
        d = np.concatenate([rng.uniform(2.0, 60.0, k - 2),
                            [edge - rng.uniform(0.0, 4.0) * ulp, edge - (slots - rng.uniform(20.0, 80.0)) * ulp,
                             edge + rng.uniform(0.0, 4.0) * ulp],
                            edge + (100.0 + 20.0 * np.arange(7)) * ulp])
        d = d[rng.permutation(d.size)]
        m = d.size
        q = np.array([*rng.uniform(-4.0, 4.0, 3), 1000.0 * i + 128.0]).astype(np.float32).astype(np.float64)
        t = 1000.0 * i + 128.0 - m + np.arange(m)
        r2 = np.maximum(d - SIG[3] * (q[3] - t) ** 2, 0.5)
        v = rng.normal(size=(m, 3))
        v *= np.sqrt(r2)[:, None] / np.linalg.norm(v, axis=1)[:, None]
        pts.append(np.concatenate([q[:3] + v / np.sqrt(SIG[:3]), t[:, None]], 1))
        off.append(off[-1] + m)
        qs.append(np.tile(q[None], (3, 1)))
    return (np.concatenate(pts).astype(np.float32), np.array(off, np.int64), np.concatenate(qs).astype(np.float32))


@pytest.mark.parametrize("k", [2, 8, 13, 32, 40, 64])
def test_distances_on_both_sides_of_a_bucket_boundary(k):
    xyzt, off, q = _clusters(k, 2500, 40 + k)
    _run(xyzt, off, q, k, SIG, K=64, what=f"bucket boundary k={k}", defer_cells=-1.0)


def _point(target):
    """(x, y) whose FP32 distance from the origin, at scales 1, is `target`."""
    target = np.float32(target)
    x = np.nextafter(np.float32(np.sqrt(float(target))), np.float32(0.0))
    while np.float32(float(x) * float(x)) > target:
        x = np.nextafter(x, np.float32(0.0))
    base = np.float32(float(x) * float(x))
    y = np.float32(np.sqrt(max(float(target) - float(base), 0.0)))
    assert np.float32(float(y) * float(y) + float(base)) == target
    return float(x), float(y)


@pytest.mark.parametrize("slots,k", [(512, 5), (1024, 33)])
def test_close_distances_two_rows_apart_are_ranked_in_fp64(slots, k):
    # A: 6 units below a bucket's start (10 of the wider ones), C: 1 above it,
    # E: at that bucket's end and listed before C.  A and C are within the
    # settlement's margin of 2^-17 (64 units), so both are ranked in FP64.
    edge = 64.0 * (1.0 + 4 * slots * 2.0 ** -23)
    u = 2.0 ** -17
    below = 6 if slots == 512 else 10
    near = [(0.125 * (i + 1), 0.0) for i in range(k - 3)]
    far = [(9.0 + i, 0.0) for i in range(6)]
    pts = near + [_point(edge - below * u), _point(edge + u), _point(edge + (slots - 1) * u)] + far
    xyzt = np.array([(x, y, 0.0, float(i)) for i, (x, y) in enumerate(pts)], np.float32)
    q = np.tile(np.array([[0.0, 0.0, 0.0, 100.0]], np.float32), (3, 1))
    st = _run(xyzt, np.array([0, len(pts)], np.int64), q, k, (1.0, 1.0, 1.0, 0.0), K=64, what="two rows apart",
              defer_cells=-1.0)
    assert st["warp_queries"] == 0
    assert st["fp64_rechecks"] == 2 * 3


def _overflow(n, seed):
    """Points and four copies of a query whose squared distances pass FP32's
    range (they are finite in FP64), scattered so that neither slot nor index
    order is the distance order."""
    rng = np.random.default_rng(seed)
    xyzt = np.zeros((n, 4), np.float32)
    xyzt[:, :2] = rng.uniform(-1e15, 1e15, (n, 2))
    xyzt[:, 3] = np.arange(n)
    return xyzt, np.tile(np.array([[3e16, -1e16, 0.0, 1e4]], np.float32), (4, 1))


@pytest.mark.parametrize("k,n", [(8, 13), (20, 40), (32, 36), (64, 90)])
def test_handed_over_queries_with_overflowed_distances(k, n):
    xyzt, q = _overflow(n, k + n)
    st = _run(xyzt, np.array([0, n], np.int64), q, k, (1e6, 1e6, 1.0, 1.0), K=10, what=f"overflow k={k} n={n}")
    assert st["warp_queries"] == 4


@pytest.mark.parametrize("k,n", [(8, 5), (20, 19), (20, 40), (64, 40)])
def test_overflowed_distances_of_a_tile(k, n):
    # ranked in FP64 also where fewer than k points exist
    xyzt, q = _overflow(n, k + n)
    for defer in (0.0, -1.0):
        _run(xyzt, np.array([0, n], np.int64), q, k, (1e6, 1e6, 1.0, 1.0), K=10, what=f"overflow k={k} n={n}",
             defer_cells=defer)


def test_spare_slots_make_no_difference_to_the_grid_order():
    # the grid order keeps lists of its own length: `extra` changes neither the
    # lists nor the work, nor what a handed-over query takes along
    wl = synth.flights(60, 80, seed=12, n_routes=5)
    ix = tnn.tnn_build_segments(torch.from_numpy(wl.xyzt).cuda(), wl.traj_off, SIG, 10)
    ref = None
    for extra in (0, 2, 4, 5, 8, 32):
        gi, gd, st = tnn.tnn_knn(ix, 12, 0.0, extra=extra, defer_cells=0.4, stats=True)
        assert st["warp_queries"] > 100
        cur = (gi, gd, st)
        if ref is None:
            ref = cur
        assert torch.equal(cur[0], ref[0]) and torch.equal(cur[1], ref[1])
        assert cur[2] == ref[2], extra


@pytest.mark.parametrize("k", [8, 16])
def test_more_queries_by_the_definition_than_warps(k):
    # every place 40 times: chains longer than the lists, so nearly every one
    # of 6,000 queries is answered by the FP64 definition
    rng = np.random.default_rng(k)
    base = np.sort(rng.uniform(0.0, 60.0, (150, 4)), axis=0)
    xyzt = np.repeat(base, 40, axis=0).astype(np.float32)
    q = xyzt.copy()
    q[:, 3] += 0.25
    st = _run(xyzt, np.array([0, 2000, 6000], np.int64), q, k, SIG, K=10, what="copies")
    assert st["exact_queries"] > 5000
