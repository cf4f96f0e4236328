"""A density that is not a number spoils the key points next to it and no others: the largest difference along a line, which
small extrema are compared with, is taken over the numbers."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


def _mask(w, sub):
    """Key points as oracle.keypoints has them, the largest |p| taken over the numbers."""
    from oracle import keypoints as K
    with np.errstate(divide="ignore", invalid="ignore"):
        rho = 1.0 / w.astype(np.float64)
    ny, nx = w.shape
    nodes = K.node_list(nx, ny, sub, sub)
    index = {nd: k for k, nd in enumerate(nodes)}
    mask = np.zeros(len(nodes), bool)
    vi, hj = set(K.line_indices(nx, sub)), set(K.line_indices(ny, sub))
    with np.errstate(invalid="ignore"):
        for orient, fixed, pts in K.lines(nx, ny, sub, sub):
            r = np.array([rho[j, i] for i, j in pts])
            for p in (r[2:] - r[:-2], (r[2:] - r[1:-1]) - (r[1:-1] - r[:-2])):
                big = np.nanmax(np.abs(p))
                for k in range(1, len(p) - 1):
                    if big == 0.0 or abs(p[k]) * 100.0 < big:
                        continue
                    if (p[k] > p[k - 1] and p[k] >= p[k + 1]) or (p[k] < p[k - 1] and p[k] <= p[k + 1]):
                        mask[index[pts[k + 1]]] = True
            for i, j in pts[1:-1]:
                if i in vi and j in hj:
                    mask[index[(i, j)]] = True
    return mask


@pytest.mark.parametrize("bad", [np.nan, 0.0, np.inf])
def test_key_points_beside_a_density_that_is_no_number(sdd, bad):
    import torch
    n = 41
    X, Y = W.identity_fields(n)
    # a bump across the lines and, far below a hundredth of it, ripples whose extrema are no key points
    w = (1.0 + np.exp(-((X - 0.4) ** 2 + (Y - 0.6) ** 2) / 0.02) + 1e-4 * np.sin(40 * X + 30 * Y)).astype(np.float32)
    clean = _mask(w, 2)
    w[20, 33] = bad
    ctx = sdd.sdd_init(n, n, 2, 2, w=torch.from_numpy(w).cuda(), xi0=torch.from_numpy(X).cuda(),
                       eta0=torch.from_numpy(Y).cuda())
    expect = _mask(w, 2)
    if np.isnan(bad):
        assert np.count_nonzero(expect != clean) <= 5 and 8 < expect.sum() < 40
    assert np.array_equal(sdd.sdd_keypoint_mask(ctx).cpu().numpy().astype(bool), expect)
