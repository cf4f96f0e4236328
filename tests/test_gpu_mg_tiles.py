"""Multigrid solves whose levels run tile by tile (subdomains beyond what one cluster holds) against sparse LU: sizes
one tile wide, tiles that end ragged, levels of one column, several systems; and direct solves repeated on a context
with other tolerances, steps and outputs against the same solves on contexts of their own."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


def _case(nx, ny):
    X, Y = W.identity_fields(nx, ny)
    w = (1.0 + 5.0 * np.exp(-((X - 0.4) ** 2 + (Y - 0.6) ** 2) / 0.03)).astype(np.float32)
    xi0, eta0 = X + 0.02 * np.sin(np.pi * X) * np.sin(2 * np.pi * Y), Y + 0.02 * np.sin(2 * np.pi * X) * np.sin(np.pi * Y)
    return w, xi0, eta0


def _ctx(sdd, nx, ny, sub_x, sub_y):
    import torch
    w, xi0, eta0 = _case(nx, ny)
    ctx = sdd.sdd_init(nx, ny, sub_x, sub_y, w=torch.from_numpy(w).cuda(), xi0=torch.from_numpy(xi0).cuda(),
                       eta0=torch.from_numpy(eta0).cuda())
    sdd.sdd_set_solver(ctx, sdd.SDD_SOLVER_MG)
    xs, ys = sdd.sdd_interface_nodes(ctx)
    vx, ve = xs + 0.03 * np.sin(7 * xs + 3 * ys), ys + 0.02 * np.cos(5 * xs)
    return ctx, torch.from_numpy(vx).cuda(), torch.from_numpy(ve).cuda()


# unknowns per subdomain: 143^2 (4.5 tiles a side, coarsest 8^2), 47 x 527 (coarsest 2 x 32), 351 x 223 (coarsest
# 10 x 6), 255^2 (coarsest 1), four of 191 x 255
@pytest.mark.parametrize("nx,ny,sub_x,sub_y", [(145, 145, 1, 1), (97, 529, 2, 1), (353, 225, 1, 1),
                                               (257, 257, 1, 1), (385, 513, 2, 2)])
def test_against_sparse_lu(sdd, nx, ny, sub_x, sub_y):
    from oracle import solver
    ctx, vx, ve = _ctx(sdd, nx, ny, sub_x, sub_y)
    gx, ge, iters = sdd.sdd_subdomain_solve(ctx, 1.5e-3, vx, ve, rtol=1e-12, max_iter=200)
    assert 0 < iters <= 30
    w, xi0, eta0 = _case(nx, ny)
    got = [gx.cpu().numpy(), ge.cpu().numpy()]
    ref = solver.subdomain_solve(w, [xi0, eta0], got, sub_x, sub_y, 1.5e-3)
    # the bound of the other multigrid solves at this tolerance
    for g, r in zip(got, ref):
        assert np.abs(g - r).max() <= 1e-9


def test_nonconvergence_is_a_status(sdd):
    # 63 x 1087 unknowns of a square domain, cells 17 times as wide as high: beyond the 30 iterations of a direct solve
    ctx, vx, ve = _ctx(sdd, 65, 1089, 1, 1)
    with pytest.raises(sdd.SddError) as e:
        sdd.sdd_subdomain_solve(ctx, 1.5e-3, vx, ve, rtol=1e-12, max_iter=200)
    assert e.value.status == sdd.SDD_ENOCONV


def test_repeated_direct_solves_keep_nothing(sdd):
    import torch
    nx, ny = 353, 225
    ctx, _, _ = _ctx(sdd, nx, ny, 1, 1)
    none = torch.empty(0, dtype=torch.float64, device="cuda")
    calls = [(1.5e-3, 1e-10, 200), (1.5e-3, 1e-6, 200), (4e-4, 1e-6, 200), (4e-4, 1e-10, 20)]
    w = _case(nx, ny)[0]
    for k, (Dt, rtol, max_iter) in enumerate(calls):
        wk = torch.from_numpy(w * np.float32(1 + k)).cuda()
        fresh, _, _ = _ctx(sdd, nx, ny, 1, 1)
        out = []
        for c in (ctx, fresh):
            sdd.sdd_set_w(c, wk)
            out.append(sdd.sdd_subdomain_solve(c, Dt, none, none, rtol=rtol, max_iter=max_iter))
        assert out[0][2] == out[1][2]
        assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
