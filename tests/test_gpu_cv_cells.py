"""The smoothed field gradients of the untrained control variate at the edges of the blocks that compute them (256
cells of a row) against the oracle's."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order", [1, 3, 33, 255])
@pytest.mark.parametrize("nx,ny", [(5, 5), (256, 6), (257, 5), (258, 7), (513, 9), (700, 5), (9, 300)])
def test_cells_match_oracle(nx, ny, order):
    import torch
    import paper_1402_0266_gb300 as sdd
    from oracle import mlp
    X, Y = W.identity_fields(nx, ny)
    xi0 = X + 0.03 * np.sin(2 * np.pi * X) * np.sin(np.pi * Y) ** 2
    eta0 = Y + 0.02 * np.sin(np.pi * X) * np.sin(3 * np.pi * Y)
    ctx = sdd.sdd_init(nx, ny, 1, 1, w=torch.ones((ny, nx), dtype=torch.float32, device="cuda"),
                       xi0=torch.from_numpy(xi0).cuda(), eta0=torch.from_numpy(eta0).cuda())
    sdd.sdd_cv_enable(ctx, sdd.SDD_CV_FIELDS)
    sdd.sdd_cv_set_fields_order(ctx, order)
    C = mlp.field_cell_gradient_table(xi0, eta0, order)[0]
    # a pass: nodes and weights rounded once, one rounding per tap, the weights add to one
    tol = 2 * (order + 3) * 2.0 ** -24 * np.abs(mlp.field_gradient_table(xi0, eta0)).max()
    assert np.abs(sdd.sdd_cv_get_cells(ctx).cpu().numpy() - C).max() <= tol
