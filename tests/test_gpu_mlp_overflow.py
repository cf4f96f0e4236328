"""A mean loss beyond the range of single precision is infinite, and the gradient beside it finite: sums over tiles keep
the errors of their additions, which an infinite sum does not have."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


# one tile of 64 rows, several to a block
@pytest.mark.parametrize("rows", [64, 64 * 700])
@pytest.mark.parametrize("size", [1e25, 1e30])
def test_gradient_and_loss_beyond_single_precision(sdd, rows, size):
    import torch
    n = 33
    X, Y = W.identity_fields(n)
    ctx = sdd.sdd_init(n, n, 2, 2, w=torch.ones((n, n), dtype=torch.float32, device="cuda"),
                       xi0=torch.from_numpy(X).cuda(), eta0=torch.from_numpy(Y).cuda())
    theta = sdd.sdd_mlp_init(ctx, 3)
    rng = np.random.default_rng(0)
    feats = torch.from_numpy(rng.standard_normal((rows, 5)).astype(np.float32)).cuda()
    norm = sdd.sdd_mlp_norm(ctx, feats)
    targets = torch.full((rows, 2), size, dtype=torch.float32, device="cuda")
    grad, loss = sdd.sdd_mlp_grad(ctx, theta, norm, feats, targets)
    # (g - y)^2 > 1e50: beyond single precision; the gradient -2 y / rows times sums of O(rows) terms of at most 1 is
    # within it
    assert bool(torch.isposinf(loss).all())
    assert bool(torch.isfinite(grad).all())
