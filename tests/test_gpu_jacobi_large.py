"""Jacobi-preconditioned solves of subdomains beyond what a cluster's registers hold, against sparse LU, on memory that
held other data before."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,sub_x,sub_y", [(200, 180, 1, 1)])
def test_against_sparse_lu(nx, ny, sub_x, sub_y):
    import torch
    import paper_1402_0266_gb300 as sdd
    from oracle import solver
    junk = torch.full((64 << 20,), 1, dtype=torch.int32, device="cuda")   # freed to the driver: reused by the context
    del junk
    torch.cuda.empty_cache()
    X, Y = W.identity_fields(nx, ny)
    w = (1.0 + 5.0 * np.exp(-((X - 0.4) ** 2 + (Y - 0.6) ** 2) / 0.03)).astype(np.float32)
    ctx = sdd.sdd_init(nx, ny, sub_x, sub_y, w=torch.from_numpy(w).cuda(), xi0=torch.from_numpy(X).cuda(),
                       eta0=torch.from_numpy(Y * Y).cuda())
    sdd.sdd_set_solver(ctx, sdd.SDD_SOLVER_JACOBI)
    xs, ys = sdd.sdd_interface_nodes(ctx)
    vx, ve = xs + 0.03 * np.sin(7 * xs + 3 * ys), ys + 0.02 * np.cos(5 * xs)
    gx, ge, iters = sdd.sdd_subdomain_solve(ctx, 1e-3, torch.from_numpy(vx).cuda(), torch.from_numpy(ve).cuda(),
                                            rtol=1e-13, max_iter=20000)
    assert 0 < iters < 20000
    got = [gx.cpu().numpy(), ge.cpu().numpy()]
    ref = solver.subdomain_solve(w, [X, Y * Y], got, sub_x, sub_y, 1e-3)
    # the bound of the other Jacobi-preconditioned solves at this tolerance
    for g, r in zip(got, ref):
        assert np.abs(g - r).max() <= 1e-9
