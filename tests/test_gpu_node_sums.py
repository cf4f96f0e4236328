"""A node's sums over its tasks and paths: one to eight warps per node in an estimate, one or four blocks per node in
the deferred scoring of a mesh step, with fewer paths than threads, ragged shares and nodes without paths."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


def _ctx(sdd, n, sub):
    import torch
    xi, eta = W.identity_fields(n)
    return sdd.sdd_init(n, n, sub, sub, w=torch.from_numpy(np.ascontiguousarray(W.w_front(n, 0.0), np.float32)).cuda(),
                        xi0=torch.from_numpy(xi).cuda(), eta0=torch.from_numpy(eta).cuda())


# tasks of 32 paths: 1 and 3 a node on average (one warp), 66, 130 and 260 (two, four and eight warps)
@pytest.mark.parametrize("paths", [1, 31, 97, 2100, 4129, 8311])
@pytest.mark.parametrize("nodes", [1, 2, 9])
def test_estimate_is_the_mean_of_its_paths(sdd, nodes, paths):
    ctx = _ctx(sdd, 33, 2)
    x, y = np.linspace(0.1, 0.8, nodes), np.full(nodes, 0.45)
    x[nodes // 2] = 0.0 if nodes > 1 else 0.3            # a node on the boundary among them
    counts = np.maximum(1, paths - 5 * np.arange(nodes))
    g = {k: v.cpu().numpy() for k, v in sdd.sdd_interface_mc_record(
        ctx, x, y, counts, dt=2e-3, Dt=1e-2, seed=5, paths_per_task=32).items()}
    first = 0
    for k in range(nodes):
        one = slice(first, first + counts[k])
        first += counts[k]
        assert g["n_exit"][k] == np.count_nonzero(g["code"][one] >= 0)
        assert g["path_steps"][k] == g["steps"][one].sum()
        if x[k] == 0.0:
            continue
        for f, start in (("xi", x[k]), ("eta", y[k])):
            d = (g["score_" + f][one] - np.float32(start)).astype(np.float32)
            S, Q = d.astype(np.float64).sum(), (d * d).astype(np.float64).sum()
            N = counts[k]
            # each lane sums its few scores in compensated single precision, off by a rounding of some scores
            assert abs(g["mean_" + f][k] - (np.float64(np.float32(start)) + S / N)) <= 1e-11
            var = max(0.0, (Q - S * S / N) / (N - 1)) if N > 1 else 0.0
            assert abs(g["se_" + f][k] ** 2 * N - var) <= 1e-10 * Q / max(N - 1, 1)


# 5, 77, 253 and 509 interface nodes: clusters of four blocks, single blocks
@pytest.mark.parametrize("n,sub", [(5, 2), (41, 2), (129, 2), (257, 2)])
@pytest.mark.parametrize("paths", [1, 7, 300, 2049])
def test_deferred_scores_match_the_step_without_deferral(sdd, n, sub, paths):
    import torch
    got = []
    for pipeline in (True, False):
        ctx = _ctx(sdd, n, sub)
        sdd.sdd_set_pipeline(ctx, pipeline)
        for k in range(2):
            sdd.sdd_set_w(ctx, torch.from_numpy(np.ascontiguousarray(W.w_front(n, 1e-3 * k), np.float32)).cuda())
            sdd.sdd_step(ctx, dt=2.5e-4, Dt=1e-3, seed=3, paths_per_node=paths)
        sdd.sdd_sync(ctx)
        got.append({k: v.cpu().numpy() for k, v in sdd.sdd_last_interface_stats(ctx).items()})
    a, b = got
    for k in ("n_exit", "path_steps"):
        assert np.array_equal(a[k], b[k])
    for k in ("mean_xi", "mean_eta", "se_xi", "se_eta"):
        # scores agree to a few units of single-precision rounding, in differently grouped sums
        assert np.abs(a[k] - b[k]).max() <= 2e-6
