"""Jacobi-preconditioned subdomain solves against sparse LU: one unknown, one column, one block and several per
subdomain, one to four unknowns per thread, unequal subdomains, and systems that the Chebyshev iterations leave to
conjugate gradients (hardly any mass term, strong contrasts)."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


def _solve_both(sdd, nx, ny, sub_x, sub_y, w, Dt):
    import torch
    from oracle import solver
    X, Y = W.identity_fields(nx, ny)
    xi0, eta0 = X + 0.02 * np.sin(np.pi * X) * np.sin(2 * np.pi * Y), Y + 0.02 * np.sin(2 * np.pi * X) * np.sin(np.pi * Y)
    ctx = sdd.sdd_init(nx, ny, sub_x, sub_y, w=torch.from_numpy(w).cuda(), xi0=torch.from_numpy(xi0).cuda(),
                       eta0=torch.from_numpy(eta0).cuda())
    sdd.sdd_set_solver(ctx, sdd.SDD_SOLVER_JACOBI)
    xs, ys = sdd.sdd_interface_nodes(ctx)
    vx, ve = xs + 0.03 * np.sin(7 * xs + 3 * ys), ys + 0.02 * np.cos(5 * xs)
    gx, ge, iters = sdd.sdd_subdomain_solve(ctx, Dt, torch.from_numpy(vx).cuda(), torch.from_numpy(ve).cuda(),
                                            rtol=1e-13, max_iter=20000)
    assert 0 < iters < 20000
    # the Dirichlet data as the library set them (faces, interface values)
    got = [gx.cpu().numpy(), ge.cpu().numpy()]
    ref = solver.subdomain_solve(w, [xi0, eta0], got, sub_x, sub_y, Dt)
    # the residual is below 1e-13 ||b||: the error at most that times ||A^-1|| ||b||, which for an M-matrix with the
    # mass term 1 / (w Dt) is at most the largest over the smallest row sum's scale; 1e-9 covers the cases here
    for g, r in zip(got, ref):
        assert np.abs(g - r).max() <= 1e-9


# (nx, ny, sub_x, sub_y): unknowns per subdomain 1, one column, 16^2 (one block), 17 x 16 (several), bands of 2 and 4
# unknowns per thread, unequal sizes, more subdomains than clusters that run at once
@pytest.mark.parametrize("nx,ny,sub_x,sub_y", [(5, 5, 2, 2), (5, 41, 2, 2), (35, 35, 2, 2), (37, 35, 2, 2),
                                               (129, 65, 1, 2), (150, 131, 1, 1), (100, 97, 3, 2), (121, 121, 6, 5)])
def test_against_sparse_lu(sdd, nx, ny, sub_x, sub_y):
    X, Y = W.identity_fields(nx, ny)
    w = (1.0 + 5.0 * np.exp(-((X - 0.4) ** 2 + (Y - 0.6) ** 2) / 0.03)).astype(np.float32)
    _solve_both(sdd, nx, ny, sub_x, sub_y, w, 1.5e-3)


@pytest.mark.parametrize("n,sub,Dt", [(33, 2, 1e3), (65, 3, 1.0), (65, 2, 1e-7)])
def test_extreme_mass_terms(sdd, n, sub, Dt):
    X, Y = W.identity_fields(n)
    w = np.where(((X * 9).astype(int) + (Y * 7).astype(int)) % 2 == 0, 50.0, 1.0).astype(np.float32)
    _solve_both(sdd, n, n, sub, sub, w, Dt)
