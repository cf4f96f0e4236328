"""Multigrid solves of two contexts from two threads: each rebuilds its graph while the other one, whose coarse levels
take another amount of shared memory, does the same."""
import threading

import numpy as np
import pytest

import workloads as W

pytestmark = pytest.mark.gpu


def test_solves_of_two_threads_do_not_disturb_each_other():
    import torch
    import paper_1402_0266_gb300 as sdd
    sdd.lib()
    jobs = []
    for n in (513, 385):   # 4 x 255^2 unknowns (63^2 and below in shared memory), 4 x 191^2 (47^2 and below)
        X, Y = W.identity_fields(n)
        w = torch.from_numpy(np.ascontiguousarray(W.w_front(n, 0.0), np.float32)).cuda()
        stream = torch.cuda.Stream()
        torch.cuda.synchronize()
        with torch.cuda.stream(stream):
            ctx = sdd.sdd_init(n, n, 2, 2, w=w, xi0=torch.from_numpy(X).cuda(), eta0=torch.from_numpy(Y).cuda(),
                               stream=stream)
            sdd.sdd_set_solver(ctx, sdd.SDD_SOLVER_MG)
            xs, ys = sdd.sdd_interface_nodes(ctx)
            a = torch.from_numpy(xs + 0.01 * np.sin(9 * ys)).cuda()
            b = torch.from_numpy(ys).cuda()
            stream.synchronize()
            ref = sdd.sdd_subdomain_solve(ctx, 1e-3, a, b)
        jobs.append((ctx, stream, a, b, ref))
    errors = []

    def work(ctx, stream, a, b, ref):
        try:
            with torch.cuda.stream(stream):
                for k in range(60):
                    # another tolerance, another graph
                    x, y, iters = sdd.sdd_subdomain_solve(ctx, 1e-3, a, b, rtol=1e-12 if k % 2 else 1e-11)
                stream.synchronize()
                assert iters == ref[2] and torch.equal(x, ref[0]) and torch.equal(y, ref[1])
        except Exception as e:   # noqa: BLE001 -- reported by the test's own thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=j) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join(120)
    assert not any(t.is_alive() for t in threads)
    assert not errors, errors
