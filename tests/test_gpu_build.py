"""Index build over the segment counts where its sorts change form (one
cluster with 1, 2 or 4 keys per thread, several launches), with tied start
times, ragged and one-point trajectories, and degenerate segments: the
exported table is in stable t_A order, its radii hold every member (and no
more than rounding above the FP64 value), and the search over its grid agrees
with the linear search."""
import numpy as np
import pytest
import torch

from paper_2112_10408_gb300 import synth
from paper_2112_10408_gb300 import tnn

pytestmark = pytest.mark.gpu
SIG = synth.SIGMA_DEFAULT


def _data(S, K, seed, ties):
    """Trajectories of 1 to 3 segments each, S in all; the last is ragged."""
    rng = np.random.default_rng(seed)
    lens, left = [], S
    while left > 0:
        s = int(min(left, rng.integers(1, 4)))
        lens.append((s - 1) * K + int(rng.integers(1, K + 1)))
        left -= s
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    n = int(off[-1])
    x = rng.uniform(0.0, 800.0, (n, 4))
    for a, b in zip(off[:-1], off[1:]):
        x[a:b, :3] = x[a, :3] + np.cumsum(rng.normal(0.0, 0.5, (b - a, 3)), 0)
        t0 = float(rng.integers(0, 6)) if ties else rng.uniform(0.0, 3000.0)
        x[a:b, 3] = t0 + 4.0 * np.arange(b - a)
    x[off[0]:off[1], :3] = x[off[0], :3]  # a segment without extent
    return x.astype(np.float32), off


def _reference(x, off, K):
    q = np.sqrt(np.array(SIG[:3]))
    p = x.astype(np.float64)
    rows = []
    for a, b in zip(off[:-1], off[1:]):
        for f in range(a, b, K):
            m = p[f:min(f + K, b)]
            A = (q * m[0, :3]).astype(np.float32).astype(np.float64)
            AB = (q * m[-1, :3] - A).astype(np.float32).astype(np.float64)
            D = q * m[:, :3] - A
            n2 = float(AB @ AB)
            lam = np.clip(D @ AB / n2, 0.0, 1.0) if n2 > 0 else np.zeros(len(m))
            rows.append((m[0, 3], m[-1, 3], f, len(m), np.sqrt(((D - lam[:, None] * AB) ** 2).sum(1).max())))
    return np.array(rows)


@pytest.mark.parametrize("ties", [False, True])
@pytest.mark.parametrize("S", [1, 2, 31, 257, 2047, 2048, 2049, 4097, 8192, 8193, 16385, 32767, 32768, 32769])
def test_segment_table_at_every_sort_form(S, ties):
    K = 3
    x, off = _data(S, K, S, ties)
    ix = tnn.tnn_build_segments(torch.from_numpy(x).cuda(), off, SIG, K)
    assert ix.n_segments == S
    seg, pm = tnn.tnn_index_export(ix)
    torch.cuda.synchronize()
    seg, pm = seg.cpu().numpy(), pm.cpu().numpy()
    ref = _reference(x, off, K)
    ref = ref[np.argsort(ref[:, 0], kind="stable")]
    assert np.array_equal(seg[:, 12].view(np.int32), ref[:, 2].astype(np.int32))
    assert np.array_equal(seg[:, 13].view(np.int32), ref[:, 3].astype(np.int32))
    assert np.array_equal(seg[:, 3], ref[:, 0].astype(np.float32))
    assert np.array_equal(pm, np.maximum.accumulate(ref[:, 1]).astype(np.float32))
    r = seg[:, 11].astype(np.float64)
    # rounded up from FP64 plus a slack of 1e-12 of the coordinates' size
    assert (r >= ref[:, 4]).all() and (r <= ref[:, 4] * (1 + 2.0 ** -22) + 2e-8).all()
    assert ix.max_radius == seg[:, 11].max()


@pytest.mark.parametrize("S,ties", [(300, True), (5000, False), (20000, True), (33000, False)])
def test_search_over_the_built_grid(S, ties):
    x, off = _data(S, 4, 7 * S, ties)
    ix = tnn.tnn_build_segments(torch.from_numpy(x).cuda(), off, SIG, 4)
    q = torch.from_numpy(x[:: max(1, len(x) // 700)].copy()).cuda()
    a = tnn.tnn_knn(ix, 10, 0.0, q=q)
    b = tnn.tnn_knn_bruteforce(ix, 10, 0.0, q=q)
    s = tnn.tnn_knn(ix, 10, 0.0, q=q, sweep=True)
    torch.cuda.synchronize()
    assert torch.equal(a[0], b[0]) and torch.equal(s[0], b[0])
    torch.testing.assert_close(a[1], b[1], rtol=1e-5, atol=0)
