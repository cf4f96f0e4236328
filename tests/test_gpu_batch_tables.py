"""The tables of a batch's instances, built together, against those of each instance alone: one to three launches of up
to sixteen grids, ragged sizes, user face data, zero maps, a density that is reported."""
import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sdd():
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    return sdd


SIZES = [(65, 65), (5, 5), (34, 33), (33, 34), (130, 35), (7, 200), (257, 129), (66, 4), (4, 66)]


def _contexts(sdd, count):
    import torch
    out = []
    for k in range(count):
        nx, ny = SIZES[k % len(SIZES)]
        X, Y = W.identity_fields(nx, ny)
        w = (1.0 + (4.0 + k) * np.exp(-((X - 0.4) ** 2 + (Y - 0.6) ** 2) / (0.01 + 0.02 * k))).astype(np.float32)
        ctx = sdd.sdd_init(nx, ny, 1, 1, w=torch.from_numpy(np.ones_like(w)).cuda(), xi0=torch.from_numpy(X).cuda(),
                           eta0=torch.from_numpy(Y * Y).cuda())
        if k % 4 == 3:
            sdd.sdd_set_boundary(ctx, torch.linspace(0.0, 1.0, sdd.faces_len(nx, ny), dtype=torch.float64, device="cuda"))
        out.append((ctx, torch.from_numpy(w).cuda()))
    return out


@pytest.mark.parametrize("count", [1, 2, 16, 17, 35])
def test_batch_matches_each_instance(sdd, count):
    together, alone = _contexts(sdd, count), _contexts(sdd, count)
    nodes = [(np.array([0.3, 0.55, 0.0]), np.array([0.6, 0.35, 0.5]), np.array([40, 33, 2])) for _ in range(count)]
    for pair in (together, alone):
        for ctx, w in pair:
            sdd.sdd_set_w(ctx, w)
    kw = dict(dt=1e-3, Dt=1e-2, seed=7)
    got = sdd.sdd_batch_interface_mc(sdd.sdd_batch_create([c for c, _ in together]), nodes, **kw)
    for k, (ctx, _) in enumerate(alone):
        one = sdd.sdd_interface_mc(ctx, *nodes[k], node_word0=3 * k, **kw)
        for name in one:
            assert (one[name].cpu().numpy() == got[k][name].cpu().numpy()).all() or \
                np.abs(one[name].cpu().numpy() - got[k][name].cpu().numpy()).max() <= 1e-12, (k, name)
        # and the zero map that the batch built, in an estimate of the instance by itself
        own = sdd.sdd_interface_mc(together[k][0], *nodes[k], node_word0=3 * k, **kw)
        for name in one:
            assert np.array_equal(one[name].cpu().numpy(), own[name].cpu().numpy()), (k, name)


def test_batch_reports_a_density(sdd):
    import torch
    ctxs = _contexts(sdd, 18)
    bad = ctxs[17][1].clone()
    bad[-1, -1] = -1.0
    sdd.sdd_set_w(ctxs[17][0], bad)
    batch = sdd.sdd_batch_create([c for c, _ in ctxs])
    nodes = [(np.array([0.3]), np.array([0.6]), np.array([8])) for _ in ctxs]
    sdd.sdd_batch_interface_mc(batch, nodes, dt=1e-3, Dt=1e-2, seed=7)
    with pytest.raises(sdd.SddError):
        sdd.sdd_batch_sync(batch)
