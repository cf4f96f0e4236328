"""max_iter bounds a Jacobi-preconditioned solve whichever of its two methods ends it: the count returned, the call's
status and the device status agree, and what conjugate gradients alone would have solved is solved."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


def _problem(sdd, m, sub, high=50.0):
    import torch
    n = sub * (m + 1) + 1
    X, Y = W.identity_fields(n)
    w = np.where(((X * 9).astype(int) + (Y * 7).astype(int)) % 2 == 0, high, 1.0).astype(np.float32)
    xi0 = X + 0.02 * np.sin(np.pi * X) * np.sin(2 * np.pi * Y)
    ctx = sdd.sdd_init(n, n, sub, sub, w=torch.from_numpy(w).cuda(), xi0=torch.from_numpy(xi0).cuda(),
                       eta0=torch.from_numpy(Y).cuda())
    sdd.sdd_set_solver(ctx, sdd.SDD_SOLVER_JACOBI)
    xs, ys = sdd.sdd_interface_nodes(ctx)
    rng = np.random.default_rng(1)
    vx, ve = xs + 0.002 * rng.standard_normal(len(xs)), ys + 0.002 * rng.standard_normal(len(xs))
    return ctx, torch.from_numpy(vx).cuda(), torch.from_numpy(ve).cuda()


def _solved(sdd, ctx, Dt, vx, ve, max_iter):
    """Solved within max_iter? The count and both statuses say the same."""
    try:
        iters = sdd.sdd_subdomain_solve(ctx, Dt, vx, ve, max_iter=max_iter)[2]
    except sdd.SddError as e:
        assert e.status == sdd.SDD_ENOCONV
        with pytest.raises(sdd.SddError) as err:
            sdd.sdd_sync(ctx)
        assert err.value.status == sdd.SDD_ENOCONV
        return False
    assert 0 <= iters <= max_iter
    sdd.sdd_sync(ctx)
    return True


# one block, clusters, one to four unknowns a thread; strong contrasts: Chebyshev iterations leave a remainder
@pytest.mark.parametrize("m,sub,Dt", [(9, 2, 0.1), (31, 2, 1e-2), (63, 2, 3e-2), (119, 2, 1e-2), (119, 3, 0.1)])
def test_statuses_and_count_agree(sdd, m, sub, Dt):
    ctx, vx, ve = _problem(sdd, m, sub)
    most = sdd.sdd_subdomain_solve(ctx, Dt, vx, ve)[2]   # iterations that no bound cuts short
    sdd.sdd_sync(ctx)
    assert not _solved(sdd, ctx, Dt, vx, ve, 3)
    for part in (0.3, 0.6, 0.8, 0.9, 0.95, 1.0, 1.05, 1.5, 1.9, 2.1, 3.0):
        _solved(sdd, ctx, Dt, vx, ve, int(part * most))


# iterations that conjugate gradients alone take for these systems: 735, 389, 853, 1903 (their number moves by a few with
# the order of the sums); the last two converge far more slowly than the Chebyshev iterations' interval says
@pytest.mark.parametrize("m,Dt,high,alone", [(119, 1e-2, 50.0, 735), (63, 1e-2, 50.0, 389), (31, 1e3, 1e4, 853),
                                             (63, 1e3, 1e4, 1903)])
def test_what_conjugate_gradients_solve_is_solved(sdd, m, Dt, high, alone):
    ctx, vx, ve = _problem(sdd, m, 2, high)
    for max_iter in (int(1.04 * alone), int(1.3 * alone), 2 * alone, 3 * alone):
        assert _solved(sdd, ctx, Dt, vx, ve, max_iter), max_iter
