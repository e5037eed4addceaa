"""Runs of passes longer than a cooperative launch may be (its barrier counts two
arrivals of every CTA and pass below a fail bit): they are cut into launches,
which changes no bits.  The limit is lowered so that a check period of 16
passes takes several launches."""
import numpy as np
import pytest
import torch

from paper_2407_19689_gb300 import instances as I
from paper_2407_19689_gb300 import pdot

pytestmark = pytest.mark.gpu


def _instance(m, n):
    ins = I.points_instance(m, n, I.seed_for(0, m + n))
    return torch.tensor(ins.C, dtype=torch.float32, device="cuda:0"), ins.f, ins.g


@pytest.mark.parametrize("m,n", [(70, 90), (1500, 1300)])
@pytest.mark.parametrize("most", [1, 5, 16])
def test_pieces_change_nothing(monkeypatch, m, n, most):
    ins = _instance(m, n)
    sols, steps, batch, launches = [], [], [], []
    for cut in (False, True):
        if cut:
            monkeypatch.setenv("PDOT_COOP_PASSES", str(most))
        s = pdot.Solver(device=0, restart_check_every=16, max_iter=96)
        sols.append(s.solve(*ins, tol=1e-9))
        X = np.outer(ins[1], ins[2]).astype(np.float32)
        n0 = s.launch_count()
        steps.append(s.pdhg_steps(*ins, X, np.zeros(m), np.zeros(n), k=16, eta=0.5 / np.sqrt(m + n)))
        launches.append(s.launch_count() - n0)
        s.close()
        B = pdot.BatchSolver(device=0, restart_check_every=16, max_iter=96, tol=1e-9)
        ids = [B.submit(*ins), B.submit(*_instance(200, 40))]
        done = B.run()
        batch.append([done[i] for i in ids])
        B.close()
    assert launches[1] - launches[0] == -(-16 // most) - 1
    for a, b in [sols] + list(zip(*batch)):
        assert a.result["passes"] == 96 and a.result["restarts"] == b.result["restarts"]
        assert torch.equal(a.X, b.X) and torch.equal(a.p, b.p) and torch.equal(a.q, b.q)
    for a, b in zip(*steps):
        assert torch.equal(a, b)
