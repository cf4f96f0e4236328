"""The training gradient over one tile, a block's several tiles and a last round that not every block has, against the
oracle's double-precision backpropagation."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows", [64, 128, 152 * 64, 153 * 64, 2 * 152 * 64 + 64])
def test_gradient_over_tiles(rows):
    import torch
    import paper_1402_0266_gb300 as sdd
    from oracle import mlp
    rng = np.random.default_rng(rows)
    feats = rng.uniform(0.0, 1.0, (rows, 5)).astype(np.float32)
    targets = (feats[:, :2] + 0.1 * rng.normal(size=(rows, 2))).astype(np.float32)
    norm = np.array([0.5] * 5 + [3.46] * 5, np.float32)
    theta = mlp.init_params(3)
    ctx = sdd.sdd_init(9, 9, 1, 1)
    block = np.zeros((2, sdd.MLP_STRIDE), np.float32)
    block[:, :theta.shape[1]] = theta
    dev = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (block.reshape(-1), norm, feats, targets)]
    grad, loss = sdd.sdd_mlp_grad(ctx, *dev)
    grad = grad.cpu().numpy().reshape(2, -1)[:, :theta.shape[1]]
    Z = mlp.normalise(feats, norm[:5].astype(np.float64), norm[5:].astype(np.float64))
    for f in range(2):
        L, g = mlp.loss_and_grad(theta[f], Z, targets[:, f])
        # single precision over tiles of 64 rows, tiles summed with their rounding errors: a few ulps of the
        # largest terms; 64-term sums of rounded tanhf and products stay well below 1e-5 in the 2-norm
        assert np.linalg.norm(grad[f] - g) <= 1e-5 * np.linalg.norm(g)
        assert abs(float(loss[f]) - L) <= 1e-5 * L
