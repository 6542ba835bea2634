"""Context features and IDW over the context sizes where the kernel changes
its mapping (ranks per lane, queries per warp) and rows that are or are not
whole 16-byte words, against float64 on the same lists."""
import numpy as np
import pytest
import torch

from paper_2112_10408_gb300 import synth
from paper_2112_10408_gb300 import tnn

pytestmark = pytest.mark.gpu
SIG = synth.SIGMA_DEFAULT


@pytest.mark.parametrize("m", [1, 3, 257])
@pytest.mark.parametrize("k", [1, 2, 4, 5, 8, 9, 15, 16, 17, 20, 31, 32, 33, 48, 63, 64])
@pytest.mark.parametrize("shift", [0, 2])
def test_features_and_idw_for_every_mapping(k, m, shift):
    wl = synth.flights(20, 50, seed=k, n_routes=3)
    ix = tnn.tnn_build_segments(torch.from_numpy(wl.xyzt).cuda(), wl.traj_off, SIG, 10)
    rng = np.random.default_rng(1000 * k + m)
    idx = rng.integers(0, wl.n, (m, k)).astype(np.int32)
    missing = rng.random((m, k)) < 0.15
    d2 = rng.uniform(0.5, 400.0, (m, k)).astype(np.float32)
    idx[missing], d2[missing] = -1, np.inf
    if m > 2:
        idx[1], d2[1] = -1, np.inf  # an empty context
    q = rng.uniform(0.0, 100.0, (m, 4)).astype(np.float32)
    mean = np.array([0.5, -0.3, 0.1, -20.0, 15.0, 3.0], np.float32)
    std = np.array([20.0, 21.0, 2.0, 30.0, 9.0, 8.0], np.float32)
    buf_i = torch.zeros(m * k + shift, dtype=torch.int32, device="cuda")
    buf_d = torch.zeros(m * k + shift, dtype=torch.float32, device="cuda")
    ti, td = buf_i[shift:].view(m, k), buf_d[shift:].view(m, k)
    ti.copy_(torch.from_numpy(idx))
    td.copy_(torch.from_numpy(d2))
    wind = torch.from_numpy(wl.wind).cuda()
    feat, idw = tnn.tnn_context_features(ix, wind, ti, td, q=torch.from_numpy(q).cuda(), mean=mean, std=std)
    only_f, none = tnn.tnn_context_features(ix, wind, ti, td, q=torch.from_numpy(q).cuda(), mean=mean, std=std,
                                            want_idw=False)
    _, only_w = tnn.tnn_context_features(ix, wind, ti, td, q=torch.from_numpy(q).cuda(), want_feat=False)
    torch.cuda.synchronize()
    assert none is None and torch.equal(only_f, feat) and torch.equal(only_w.nan_to_num(-1), idw.nan_to_num(-1))
    j = np.where(idx >= 0, idx, 0)
    p, w = wl.xyzt.astype(np.float64)[j], wl.wind.astype(np.float64)[j]
    f = np.concatenate([(p - q[:, None]) * np.sqrt(np.array(SIG)), w], 2)
    f = np.where((idx >= 0)[..., None], (f - mean.astype(np.float64)) / std, 0.0).reshape(m, 6 * k)
    got = feat.float().cpu().numpy()
    # BF16 rounding (2^-9 relative) plus FP32 arithmetic on values up to 2000
    np.testing.assert_allclose(got, f, rtol=2.0 ** -8, atol=1e-3)
    wt = np.where(idx >= 0, 1.0 / (d2.astype(np.float64) + 1e-6), 0.0)
    with np.errstate(invalid="ignore"):
        ref = (wt[..., None] * w).sum(1) / wt.sum(1)[:, None]
    np.testing.assert_allclose(idw.cpu().numpy(), ref, rtol=1e-5, atol=1e-5)
