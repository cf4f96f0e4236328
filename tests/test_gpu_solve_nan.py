"""A value that is not a number among a solve's inputs is reported as a solve that did not converge, by every solver: in
the call that returns iteration counts, and at the next synchronisation."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


# Jacobi: 16^2 unknowns (one block), 19^2 and 63^2 (clusters), 199^2 (beyond their registers); multigrid in one cluster and
# as a chain of launches; direct
@pytest.mark.parametrize("solver,n", [("JACOBI", 35), ("JACOBI", 41), ("JACOBI", 129), ("JACOBI", 401), ("MG", 257),
                                      ("MG", 513), ("DIRECT", 41)])
@pytest.mark.parametrize("where", ["interface", "field"])
def test_not_a_number_is_reported(sdd, solver, n, where):
    import torch
    X, Y = W.identity_fields(n)
    w = torch.from_numpy(np.ascontiguousarray(W.w_front(n, 0.0), np.float32)).cuda()
    xi0 = X.copy()
    if where == "field":
        xi0[n // 4, n // 5] = np.nan
    ctx = sdd.sdd_init(n, n, 2, 2, w=w, xi0=torch.from_numpy(xi0).cuda(), eta0=torch.from_numpy(Y).cuda())
    sdd.sdd_set_solver(ctx, getattr(sdd, "SDD_SOLVER_" + solver))
    xs, ys = sdd.sdd_interface_nodes(ctx)
    ve = ys.copy()
    if where == "interface":
        ve[len(ve) // 3] = np.nan
    a, b = torch.from_numpy(xs).cuda(), torch.from_numpy(ve).cuda()
    with pytest.raises(sdd.SddError) as err:
        sdd.sdd_subdomain_solve(ctx, 1e-3, a, b)
    assert err.value.status == sdd.SDD_ENOCONV
    with pytest.raises(sdd.SddError):
        sdd.sdd_sync(ctx)   # the status of the call before
    sdd.sdd_subdomain_solve(ctx, 1e-3, a, b, want_iters=False)
    with pytest.raises(sdd.SddError) as err:
        sdd.sdd_sync(ctx)
    assert err.value.status == sdd.SDD_ENOCONV
    # the context is usable afterwards
    sdd.sdd_set_fields(ctx, torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda())
    gx, _, iters = sdd.sdd_subdomain_solve(ctx, 1e-3, a, torch.from_numpy(ys).cuda())
    assert 0 < iters < 20000 and bool(torch.isfinite(gx).all())
    sdd.sdd_sync(ctx)
