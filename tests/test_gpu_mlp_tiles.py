"""The estimator's gradient at the edges of its 32-sample tiles: a full tile, one sample less,
and more samples than the partial sums hold tiles (several tiles to a CTA, the last one ragged)."""

import numpy as np
import pytest
import torch

import oracle as O

pytestmark = pytest.mark.gpu
cuda = pytest.mark.skipif(not torch.cuda.is_available(), reason="needs a CUDA GPU")
M = O.mlp_oracle
F, H = 8, 64
# float sums of at most 64 (a layer) + 64 (a CTA's samples) + 128 + 8 (partials) terms: 264 roundings
# of 6e-8, four times for the layers they pass through; the targets' offset keeps the sums from cancelling
TOL = 1e-4


@cuda
@pytest.mark.parametrize("n", [31, 32, 36007])
def test_gradient_of_whole_and_ragged_tiles(n):
    from paper_2201_06958_gb300 import build_lib, tdb
    build_lib.build()
    rng = np.random.default_rng(4100 + n)
    th = (M.init_params(F, H, rng) + 0.05 * rng.standard_normal(M.n_params(F, H))).astype(np.float32)
    X = rng.standard_normal((n, F)).astype(np.float32)
    t = (3.0 + rng.standard_normal(n)).astype(np.float32)
    d = lambda a: torch.from_numpy(a).cuda()
    loss, grad = tdb.mlp_loss_grad(d(th), d(X), d(t))
    L_ref, g_ref = M.loss_and_grad(th.astype(np.float64), X.astype(np.float64), t.astype(np.float64), F, H)
    assert abs(loss.item() - L_ref) <= TOL * L_ref
    g = grad.cpu().numpy().astype(np.float64)
    assert np.linalg.norm(g - g_ref) <= TOL * np.linalg.norm(g_ref)
