"""Batches long enough that a warp of the GKA-MLP gradient takes several
queries and a CTA of the context features several rounds of its pipeline."""
import numpy as np
import pytest
import torch

from oracle import nowcast as nc
from paper_2112_10408_gb300 import tnn
from tests import test_gpu_features as features
from tests import test_gpu_nowcast as nowcast

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [4864, 5001, 20003])  # one query per warp up to 4,864
def test_gkamlp_gradient_of_several_queries_per_warp(B):
    wl, ix, idx, wind = nowcast._gka_setup()
    idx_h = idx.cpu().numpy()
    full = np.nonzero((idx_h >= 0).all(axis=1))[0].astype(np.int32)
    rows = full[np.random.default_rng(B).integers(0, full.size, B)]  # rows may repeat
    H = 8
    g = tnn.GKAMLP((0.05, 4.0, 1e-4), hidden=H, seed=5)
    w, _ = g.get_params()
    w[4 * H:7 * H] = (0.3 * np.random.default_rng(6).normal(size=3 * H)).astype(np.float32)
    g.set_params(w)
    loss, grad = g.gradients(ix, wind, torch.from_numpy(rows).cuda(), idx)
    rl, rg = nc.gkamlp_loss_grad(wl.xyzt, wl.wind, rows, idx_h, w, H, wl.xyzt.min(axis=0), wl.xyzt.max(axis=0))
    assert float(loss.item()) == pytest.approx(rl, rel=1e-4)
    np.testing.assert_allclose(grad.cpu().numpy(), rg, rtol=5e-3, atol=2e-3 * np.abs(rg).max())


@pytest.mark.parametrize("m", [20011, 50003])
@pytest.mark.parametrize("k", [20, 32, 33, 64])
def test_features_and_idw_of_several_rounds(k, m):
    features.test_features_and_idw_for_every_mapping(k, m, 0)
