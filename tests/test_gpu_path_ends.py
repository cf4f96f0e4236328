"""A path's record does not depend on the lanes around it: paths that leave early wait in their lane for others before
they are scored and replaced, so tasks of one path, of a warp's paths and of many give the same records."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


@pytest.mark.parametrize("exit_mode,cv", [(0, False), (1, False), (2, False), (0, True), (1, True)])
@pytest.mark.parametrize("K", [1, 7, 24])
def test_records_whatever_the_task(sdd, exit_mode, cv, K):
    import torch
    nx, ny = 65, 49
    X, Y = W.identity_fields(nx, ny)
    w = (1.0 + 5.0 * np.exp(-((X - 0.4) ** 2 + (Y - 0.6) ** 2) / 0.03)).astype(np.float32)
    ctx = sdd.sdd_init(nx, ny, 1, 1, w=torch.from_numpy(w).cuda(), xi0=torch.from_numpy(X + 0.05 * X * Y).cuda(),
                       eta0=torch.from_numpy(Y - 0.04 * X * X).cuda())
    if cv:
        sdd.sdd_cv_enable(ctx, sdd.SDD_CV_FIELDS)
    # starts next to a face, a corner and inside: all, most and a few of the paths leave
    x, y = np.array([0.01, 0.98, 0.5, 0.12]), np.array([0.4, 0.03, 0.5, 0.6])
    counts = np.array([1, 700, 333, 1025])
    kw = dict(dt=1e-3, Dt=1e-3 * K, seed=11, exit_mode=exit_mode)
    got = [{k: v.cpu().numpy() for k, v in sdd.sdd_interface_mc_record(ctx, x, y, counts, paths_per_task=t, **kw).items()}
           for t in (32, 96, 2048)]
    assert (got[0]["code"] >= 0).any() and (K == 1 or (got[0]["code"] < 0).any())
    for g in got[1:]:
        for k in ("steps", "code", "score_xi", "score_eta", "x_end", "y_end", "n_exit", "path_steps"):
            assert np.array_equal(got[0][k], g[k]), k
