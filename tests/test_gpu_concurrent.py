"""Handles in use at the same time: solves and batches whose cooperative launches
each want most of the device, from several threads on streams of their own,
give what they give alone."""
import threading

import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import instances as I
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


def _instance(m, n):
    ins = I.points_instance(m, n, I.seed_for(0, m + n))
    return torch.tensor(ins.C, dtype=torch.float32, device="cuda:0"), ins.f, ins.g


def _solve(ins):
    s = pdot.Solver(device=0, max_iter=320, time_limit_s=60.0)
    sol = s.solve(*ins, tol=1e-9)
    s.close()
    return [sol.X, sol.p, sol.q]


def _steps(ins):
    m, n = ins[0].shape
    s = pdot.Solver(device=0)
    out = s.pdhg_steps(*ins, np.outer(ins[1], ins[2]).astype(np.float32), np.zeros(m), np.zeros(n), k=200,
                       eta=0.5 / np.sqrt(m + n))
    s.close()
    return list(out)


def _batch(ins):
    B = pdot.BatchSolver(device=0, max_iter=320, tol=1e-9)
    ids = [B.submit(*i) for i in ins]
    done = B.run()
    out = [t for i in ids for t in (done[i].X, done[i].p, done[i].q)]
    B.close()
    return out


def test_threads_give_the_same_as_alone():
    jobs = [(_solve, _instance(2300, 2200)), (_steps, _instance(1500, 1300)),
            (_batch, [_instance(m, n) for m, n in ((900, 1100), (64, 64), (700, 300))])]
    streams = [torch.cuda.Stream() for _ in jobs]
    torch.cuda.synchronize()

    def run(j):   # (a solver takes the current stream)
        fn, ins = jobs[j]
        with torch.cuda.stream(streams[j]):
            return fn(ins)

    alone = [run(j) for j in range(len(jobs))]
    got = [[None] * 3 for _ in jobs]

    def work(j):
        for r in range(3):
            got[j][r] = run(j)

    threads = [threading.Thread(target=work, args=(j,)) for j in range(len(jobs))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for want, runs in zip(alone, got):
        for out in runs:
            assert len(out) == len(want) and all(torch.equal(a, b) for a, b in zip(out, want))
