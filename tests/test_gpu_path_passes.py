"""The path kernels' passes over sub-step pairs: path counts around a warp's 32 lanes, odd and single
sub-steps, refills of lanes whose paths left, starts next to the boundary, and the grid size from which
single contexts run the batch kernels."""
import numpy as np
import pytest

import workloads as W
from tests import _parity as PT

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


@pytest.fixture(scope="module")
def oracle_mod():
    import oracle
    oracle.build()
    return oracle


def _np(d):
    return {k: v.cpu().numpy() for k, v in d.items()}


def _ctx(sdd, w, xi, eta):
    import torch
    ny, nx = w.shape
    return sdd.sdd_init(nx, ny, 2, 2, w=torch.from_numpy(w).cuda(), xi0=torch.from_numpy(xi).cuda(),
                        eta0=torch.from_numpy(eta).cuda())


# K = 1: a pair without its second sub-step; 2: one full pair; 3, 7: odd; 40: many passes
@pytest.mark.parametrize("K", [1, 2, 3, 7, 40])
@pytest.mark.parametrize("exit_mode", [0, 1])
def test_records_at_lane_and_pair_edges(sdd, oracle_mod, K, exit_mode):
    nx, ny = 37, 23
    X, Y = W.identity_fields(nx, ny)
    w = (1.0 + 4.0 * np.exp(-((X - 0.6) ** 2 + (Y - 0.4) ** 2) / 0.02)).astype(np.float32)
    # a cell away from the boundary (most paths leave: refills), one float off it, and the middle
    xs = np.array([1.0 / (nx - 1), 0.5, 1.0 - 2.0 ** -25, 0.5, 0.999, 0.4])
    ys = np.array([0.5, 1.0 / (ny - 1), 0.5, 0.5, 0.999, 0.7])
    npaths = np.array([1023, 1, 31, 32, 33, 450])
    kw = dict(dt=1e-3, Dt=K * 1e-3, seed=77, step_index=3, exit_mode=exit_mode)
    g = _np(sdd.sdd_interface_mc_record(_ctx(sdd, w, X, Y), xs, ys, npaths, paths_per_task=128, **kw))
    o = oracle_mod.interface_mc(oracle_mod.Problem(w, X, Y), xs, ys, npaths, record=True, **kw)
    same, _ = PT.assert_records(g, o)
    PT.assert_nodes(g, o, npaths, same, np.concatenate([[0], np.cumsum(npaths)]))


@pytest.mark.parametrize("n", [2897, 2898])   # 2896^2 cells take the single-instance kernels, 2897^2 the batch ones
def test_records_around_the_largest_single_instance_grid(sdd, oracle_mod, n):
    X, Y = W.identity_fields(n)
    w = W.w_ring(n, 0.1)
    xs, ys = np.array([0.5, 0.999, 0.2]), np.array([0.2, 0.999, 0.5])
    kw = dict(dt=1e-6, Dt=1e-5, seed=5, step_index=1)
    g = _np(sdd.sdd_interface_mc_record(_ctx(sdd, w, X, Y), xs, ys, 200, **kw))
    o = oracle_mod.interface_mc(oracle_mod.Problem(w, X, Y), xs, ys, 200, record=True, **kw)
    PT.assert_records(g, o)


@pytest.mark.parametrize("nx,ny", [(5, 9), (47, 48), (48, 95), (300, 61)])
def test_zero_map_marks_every_tile_with_drift(sdd, nx, ny):
    # grids coarser and finer than the map's tiles, drift in a narrow part of the square: the records
    # with the map are those without it, bit for bit
    X, Y = W.identity_fields(nx, ny)
    w = np.where((X > 0.3) & (X < 0.55) & (Y < 0.6), 1.0 + X * Y, 1.0).astype(np.float32)
    ctx = _ctx(sdd, w, X, Y)
    rng = np.random.default_rng(nx)
    xs, ys = rng.uniform(0.02, 0.98, 40), rng.uniform(0.02, 0.98, 40)
    kw = dict(dt=5e-4, Dt=1e-2, seed=8)
    a = _np(sdd.sdd_interface_mc_record(ctx, xs, ys, 500, zero_map=1, **kw))
    b = _np(sdd.sdd_interface_mc_record(ctx, xs, ys, 500, zero_map=2, **kw))
    for k in a:
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
