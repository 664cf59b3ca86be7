"""GPU checks of the training kernel (xg_mlp_loss_grad) against the float64
oracle at the edges of its chunks and blocks: a single sample, a chunk less and
more one, several chunks per block, and the smallest leading dimension."""

import numpy as np
import pytest

from oracle import closure as OC

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 31, 32, 33, 4097, 10001, 40000])
def test_loss_and_gradient_sizes(cuda_device, n):
    import torch
    from paper_2504_08157_gb300 import xg
    r = np.random.RandomState(n)
    p = (r.uniform(-1, 1, xg.XG_CLOSURE_PARAMS) / 8).astype(np.float32)
    X = r.randn(21, n).astype(np.float32)
    T = r.randn(5, n).astype(np.float32)
    mean, scale = (0.1 * r.randn(21)).astype(np.float32), r.uniform(0.5, 2, 21).astype(np.float32)
    out = r.uniform(0.5, 2, 5).astype(np.float32)
    t = lambda a: torch.from_numpy(a).to(cuda_device)
    g = torch.empty(xg.XG_CLOSURE_PARAMS, dtype=torch.float32, device=cuda_device)
    loss = xg.xg_mlp_loss_grad(t(p), t(X), t(T), t(mean), t(scale), t(out), g)
    Z = np.clip((X.astype(np.float64) - mean[:, None]) * scale[:, None], -8, 8)
    ref, rg = OC.loss_and_grad(p.astype(np.float64), Z.T, (T.astype(np.float64) / out[:, None]).T)
    assert abs(loss - ref) <= 1e-5 * ref
    assert np.linalg.norm(g.cpu().numpy() - rg) <= 1e-5 * np.linalg.norm(rg)
