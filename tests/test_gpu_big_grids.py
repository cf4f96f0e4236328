"""Grids of more than 2^23 cells: a single context's path kernels (integer cell index, tables as parameters, zero map)
against the batch kernels, the oracle, and themselves without the map."""
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


def _problem(nx, ny):
    X, Y = W.identity_fields(nx, ny)
    w = np.where((X > 0.3) & (X < 0.55) & (Y < 0.6), 1.0 + X * Y, 1.0).astype(np.float32)   # drift in a part
    return w, X + 0.02 * np.sin(2 * np.pi * X) * np.sin(np.pi * Y), Y + 0.02 * np.sin(3 * np.pi * X) * np.sin(np.pi * Y)


XS = np.array([0.31, 0.5, 0.9995, 0.2, 0.548, 0.3001])
YS = np.array([0.2, 0.599, 0.9995, 0.5, 0.1, 0.0004])
COUNTS = np.array([300, 33, 200, 1, 32, 257])


# the last grid below the line, the first above it, and a long one above it
@pytest.mark.parametrize("nx,ny", [(2897, 2897), (2898, 2898), (8200, 1100)])
def test_single_context_is_a_batch_of_one(sdd, nx, ny):
    w, xi, eta = _problem(nx, ny)
    ctx = _ctx(sdd, w, xi, eta)
    batch = sdd.sdd_batch_create([ctx])
    for mode, K in ((0, 1), (0, 8), (0, 9), (1, 6)):
        kw = dict(dt=2e-6, Dt=2e-6 * K, seed=4, exit_mode=mode, paths_per_task=64)
        b = _np(sdd.sdd_batch_interface_mc(batch, [(XS, YS, COUNTS)], **kw)[0])
        for zero_map in (1, 2):
            a = _np(sdd.sdd_interface_mc(ctx, XS, YS, COUNTS, zero_map=zero_map, **kw))
            for k in a:
                # the same scores, in sums over the same lanes and tasks
                np.testing.assert_array_equal(a[k], b[k], err_msg=f"{mode} {K} {k}")
        on = _np(sdd.sdd_interface_mc_record(ctx, XS, YS, COUNTS, zero_map=1, **kw))
        off = _np(sdd.sdd_interface_mc_record(ctx, XS, YS, COUNTS, zero_map=2, **kw))
        for k in on:
            np.testing.assert_array_equal(on[k], off[k], err_msg=f"{mode} {K} {k}")


@pytest.mark.parametrize("nx,ny", [(2898, 2898), (8200, 1100)])
@pytest.mark.parametrize("cv", ["fields", "table"])
def test_control_variate_records_match_oracle(sdd, oracle_mod, nx, ny, cv):
    import torch
    from oracle import mlp
    w, xi, eta = _problem(nx, ny)
    ctx = _ctx(sdd, w, xi, eta)
    if cv == "fields":
        sdd.sdd_cv_enable(ctx, sdd.SDD_CV_FIELDS)
        sdd.sdd_cv_set_fields_order(ctx, 1)
        T = mlp.field_cell_gradient_table(xi, eta, 1)
    else:
        T = mlp.field_gradient_table(xi, eta)
        sdd.sdd_cv_set_table(ctx, torch.from_numpy(np.ascontiguousarray(T)).cuda())
        sdd.sdd_cv_enable(ctx, sdd.SDD_CV_TABLE)
    for mode in (0, 1):
        kw = dict(dt=2e-6, Dt=1.4e-5, seed=11, exit_mode=mode)
        o = oracle_mod.interface_mc(oracle_mod.Problem(w, xi, eta), XS, YS, COUNTS, record=True,
                                    cv_table=np.ascontiguousarray(T), **kw)
        for zero_map in (1, 2):
            g = _np(sdd.sdd_interface_mc_record(ctx, XS, YS, COUNTS, zero_map=zero_map, **kw))
            # a table's half-precision corners are off by 2^-11 of a gradient near 1, times increments that add up to
            # a few sqrt(2 Dt) = 0.005
            PT.assert_records(g, o)


def test_the_tuner_finds_the_zero_map(sdd):
    # no drift anywhere: the launch with the map reads no drift record, the one without reads one every sub-step
    nx = ny = 2900
    X, Y = W.identity_fields(nx, ny)
    ctx = _ctx(sdd, np.ones((ny, nx), np.float32), X, Y)
    xs, ys = np.random.default_rng(0).uniform(0.2, 0.8, (2, 400))
    shape = sdd.sdd_autotune(ctx, xs, ys, np.full(400, 8000), dt=1e-5, Dt=1e-3)
    assert shape["zero_map"] == 1


def test_deferred_scores_match_the_step_without_deferral(sdd):
    import torch
    n, sub = 2945, 23   # 529 subdomains of 127^2 unknowns: one launch solves them, so the step can defer its scores
    X, Y = W.identity_fields(n)
    got = []
    for pipeline in (True, False):
        ctx = sdd.sdd_init(n, n, sub, sub, w=torch.from_numpy(W.w_ring(n, 0.0)).cuda(), xi0=torch.from_numpy(X).cuda(),
                           eta0=torch.from_numpy(Y).cuda())
        sdd.sdd_set_pipeline(ctx, pipeline)
        for k in range(2):
            sdd.sdd_set_w(ctx, torch.from_numpy(W.w_ring(n, 1e-3 * k)).cuda())
            sdd.sdd_step(ctx, dt=2e-6, Dt=1e-5, seed=3, paths_per_node=7)
            assert sdd.sdd_pipeline_in_use(ctx) == pipeline
        sdd.sdd_sync(ctx)
        got.append(_np(sdd.sdd_last_interface_stats(ctx)))
        del ctx
    a, b = got
    for k in ("n_exit", "path_steps"):
        np.testing.assert_array_equal(a[k], b[k], err_msg=k)
    for k in ("mean_xi", "mean_eta", "se_xi", "se_eta"):
        # scores agree to a few units of single-precision rounding, in differently grouped sums
        assert np.abs(a[k] - b[k]).max() <= 2e-6, k
