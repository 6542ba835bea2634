"""Index builds near the largest sizes: the exported table of segments is that
of the points to their end, and a search finds the neighbours there.  Skipped
where the device or the host has too little memory left."""
import numpy as np
import pytest
import torch

from paper_2112_10408_gb300 import tnn

pytestmark = pytest.mark.gpu
CHUNK = 1 << 26


def _need(device_gb, host_gb):
    torch.cuda.empty_cache()
    tnn.tnn_memory_trim()
    host = next(int(ln.split()[1]) for ln in open("/proc/meminfo") if ln.startswith("MemAvailable")) >> 20
    if torch.cuda.mem_get_info()[0] < device_gb << 30 or host < host_gb:
        pytest.skip(f"needs {device_gb} GB of device memory and {host_gb} GB of host memory")


def _points(n):
    """Point i: x = i mod 256, t = i div 256 (t + 1/2 is exact in FP32)."""
    x = torch.zeros((n, 4), device="cuda")
    for a in range(0, n, CHUNK):
        i = torch.arange(a, min(n, a + CHUNK), device="cuda")
        x[a:a + CHUNK, 0] = (i & 255).float()
        x[a:a + CHUNK, 3] = (i >> 8).float()
    return x


def _check_search(ix, rows):
    """Nearest of (x + 1/4, t + 1/2) at unit scales: the point itself, the
    next, the one before, the one a second earlier."""
    rows = np.asarray(rows, np.int64)
    assert ((rows & 255) >= 1).all() and ((rows & 255) <= 254).all()
    q = np.zeros((rows.size, 4), np.float32)
    q[:, 0], q[:, 3] = (rows & 255) + 0.25, (rows >> 8) + 0.5
    idx, d2 = tnn.tnn_knn(ix, 4, 0.0, q=torch.from_numpy(q).cuda())
    assert idx.cpu().numpy().tolist() == [[r, r + 1, r - 1, r - 256] for r in rows.tolist()]
    assert d2.cpu().numpy().tolist() == [[0.3125, 0.8125, 1.8125, 2.3125]] * rows.size


@pytest.mark.parametrize("n,K,length,device_gb", [((1 << 31) - 65, 64, 1 << 15, 130),
                                                  ((1 << 30) + 4, 2, 1 << 10, 215)])  # 2^29 + 2 segments
def test_points_up_to_the_limit(n, K, length, device_gb):
    _need(device_gb, 8)
    x = _points(n)
    off = np.append(np.arange(0, n, length), n).astype(np.int64)
    ix = tnn.tnn_build_segments(x, off, (1.0, 1.0, 1.0, 1.0), K)
    S = -(-n // K)
    assert ix.n_segments == S
    seg, pm = tnn.tnn_index_export(ix)
    s = torch.arange(S, device="cuda")
    first = seg[:, 12].contiguous().view(torch.int32)
    # 256 / K segments begin with every second: t_A order is the build order
    assert torch.equal(first, (K * s).int())
    count = seg[:, 13].contiguous().view(torch.int32)
    assert bool((count[:-1] == K).all()) and int(count[-1]) == n - K * (S - 1)
    assert torch.equal(seg[:, 3], ((K * s) >> 8).float()) and torch.equal(pm, seg[:, 7])
    last = torch.clamp(K * s + K - 1, max=n - 1)
    assert torch.equal(seg[:, 7], (last >> 8).float())
    assert torch.equal(seg[:, 0], ((K * s) & 255).float())
    _check_search(ix, [n - 10, n - 200, (1 << 29) + 77, (1 << 20) + 50, 130 * 256 + 5, 2 * 256 + 66])
    del x, seg, pm, s, first, count, last
    ix.destroy()
    tnn.tnn_memory_trim()
    torch.cuda.empty_cache()


def test_tens_of_millions_of_one_point_trajectories():
    n = 65_700_000
    _need(40, 8)
    x = _points(n)
    x[:, 3] = (torch.arange(n, device="cuda") * 7919 % (1 << 20)).float()  # in no order, with ties
    off = np.arange(n + 1, dtype=np.int64)
    ix = tnn.tnn_build_segments(x, off, (1.0, 1.0, 1.0, 1.0), 2)
    assert ix.n_segments == n
    seg, pm = tnn.tnn_index_export(ix)
    t, first = torch.sort(x[:, 3], stable=True)
    assert torch.equal(seg[:, 12].contiguous().view(torch.int32), first.int())
    assert bool((seg[:, 13].contiguous().view(torch.int32) == 1).all())
    assert torch.equal(seg[:, 3], t) and torch.equal(pm, t)
    del x, seg, pm, t, first
    ix.destroy()
    tnn.tnn_memory_trim()
    torch.cuda.empty_cache()
